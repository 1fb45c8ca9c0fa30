// D3Q19 step with the populations stored as 16-bit offsets from their
// equilibria (FP16 or BF16), arithmetic in FP32.
//
// A post-collision value is stored as
//     f*_i(x) = f_i^eq(M(x)) + s_f h_i(x),   g*_i(x) = g_i^eq(M(x)) + s_g k_i(x),
// where M(x) = (phi, mu, p, u) are the FP32 macroscopic fields of node x from
// the same collision, f^eq is Eq. H_i, g^eq the equilibrium of Eq. G_i (with
// s_i(u)), h and k are 16-bit numbers and s_f, s_g are per-field scales
// (powers of two).  Only the non-equilibrium part and the source, which are
// small, pass through the 16-bit rounding.  Pull layout as in the other
// precisions: f*_i(x) is stored at x, the step at y reads it from y - c_i
// together with the macros of y - c_i.
//
// Storage of one parity of the double buffer (offset_layout):
//   f buffer: h[19][N] (u16) | M[7][N] (FP32: phi, mu, p, ux, uy, uz, B) | s_f, s_g
//   g buffer: k[19][N] (u16)
// B = phi + alpha sum_{i != 0} w_i (mu(x + c_i) - mu(x)) is the part of the
// next step's phi(x) that does not depend on the offsets; the step writes it
// from its mu ring, so the next phi pass streams B and the offsets only.
// The rest population keeps phi exactly the way the FP32 path's compensated
// pair does: phi (FP32) in M is its high word, and the rounding residual of
// phi is folded into the rest offset h_0.
//
// Scales: a step reads the scales stored with its source buffer and writes
// with the context's target scales, which it also stores with the
// destination buffer.  off_refresh (run with the diagnostics) sets the
// targets from the largest stored offsets: max |offset| / s near 2^12 (FP16
// range 65504), never below 2^-16 (so no offset up to about 1 can overflow
// between two refreshes).
//
// A step is two passes, as in the FP32 D3Q19 path: d3q19_off_phi_kernel
// writes phi from the pulled populations, then d3q19_off_pass_kernel marches
// down z with phi, mu and the macro planes of the source state in
// shared-memory rings.  HBM traffic per node: 38 + 4 + 4 B (pass 1) and
// 38 + 38 + 24 + 4 + 4 B read, 38 + 38 + 28 + 4 B written (pass 2).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <float.h>
#include <math.h>

#include "d3q19_lattice.cuh"
#include "launch.cuh"
#include "lbm_internal.h"
#include "pair32.cuh"

namespace wblbm {
namespace {

using namespace d3;

struct CodecF16 {
    static constexpr unsigned short INF_BITS = 0x7c00;
    __device__ static float dec(unsigned short u) { return __half2float(__ushort_as_half(u)); }
    __device__ static unsigned short enc(float v) { return __half_as_ushort(__float2half_rn(v)); }
    // two values in one word, the first in the low half
    __device__ static float2 dec2(unsigned v)
    {
        return __half22float2(*reinterpret_cast<const __half2 *>(&v));
    }
    __device__ static unsigned enc2(float2 v)
    {
        const __half2 h = __float22half2_rn(v);
        return *reinterpret_cast<const unsigned *>(&h);
    }
};
struct CodecBF16 {
    static constexpr unsigned short INF_BITS = 0x7f80;
    __device__ static float dec(unsigned short u)
    {
        return __bfloat162float(__ushort_as_bfloat16(u));
    }
    __device__ static unsigned short enc(float v)
    {
        return __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
    __device__ static float2 dec2(unsigned v)
    {
        return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
    }
    __device__ static unsigned enc2(float2 v)
    {
        const __nv_bfloat162 h = __float22bfloat162_rn(v);
        return *reinterpret_cast<const unsigned *>(&h);
    }
};

// views of one parity of the offset storage
struct OffBuf {
    unsigned short *h, *k;  // f and g offsets [19][N]
    float *M;               // macros [7][N] (phi, mu, p, u, B)
    float *sc;              // s_f, s_g
};

__host__ __device__ inline OffBuf off_view(const void *fbuf, const void *gbuf, long long N)
{
    const OffsetLayout L = offset_layout(N, 19, 3);  // 3 + 4 FP32 arrays
    char *fb = (char *)fbuf;
    return OffBuf{(unsigned short *)fb, (unsigned short *)gbuf, (float *)(fb + L.mac_off),
                  (float *)(fb + L.sc_off)};
}

// ------------------------------------------------------------------ pass 1
// phi(x) = sum_i f_i(x): the rest value phi(x) - (1 - w0) alpha mu(x) + s_f h_0(x)
// and the moving values w_i alpha mu(x - c_i) + s_f h_i(x - c_i), i.e.
// B(x) + s_f sum_i h_i(x - c_i) with B = phi + alpha sum_{i != 0} w_i (mu(x - c_i) - mu(x)).
// grid (ceil(nx / PHI_TX), ny, nz): one thread per node of a row
constexpr int PHI_TX = 128;
template <class C>
__global__ void __launch_bounds__(PHI_TX)
    d3q19_off_phi_kernel(const StepParams<float> P, const OffBuf src, float *__restrict__ phi)
{
    const int bx = pdl_wait(blockIdx.x);
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x = bx * PHI_TX + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= nx) return;
    const unsigned N = (unsigned)P.N;
    const Nb b = make_nb(x, y, z, nx, ny, nz);
    const unsigned n = b.at(0, 0, 0);
    float sh = C::dec(__ldg(src.h + n));
#pragma unroll
    for (int i = 1; i < 19; ++i) sh += C::dec(__ldg(src.h + (i * N + b.at(-c3x(i), -c3y(i), -c3z(i)))));
    phi[n] = __ldg(src.M + 6 * N + n) + __ldg(after_wait(src.sc)) * sh;
}

// B(x) from stored macros (after an initial condition or a state exchange)
__global__ void d3q19_off_prep_k(const StepParams<float> P, OffBuf o)
{
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x = blockIdx.x * PHI_TX + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= nx) return;
    const unsigned N = (unsigned)P.N;
    const Nb b = make_nb(x, y, z, nx, ny, nz);
    const unsigned n = b.at(0, 0, 0);
    const float *mu = o.M + N, mux = mu[n];
    float dfa = 0.0f, ded = 0.0f;
    for (int i = 1; i < 19; ++i) {
        const float d = mu[b.at(c3x(i), c3y(i), c3z(i))] - mux;
        if (i <= 6)
            dfa += d;
        else
            ded += d;
    }
    o.M[6 * N + n] = o.M[n] + P.alpha * (1.0f / 18.0f * dfa + 1.0f / 36.0f * ded);
}

// ------------------------------------------------------------------ pass 2

// One CTA's diagnostics partial from its NT threads' values (all of them call it)
template <int NT>
__device__ __forceinline__ void off_partial(int tid, double d_phi, double d_E, double d_u2,
                                            double d_mumin, double d_mumax, double d_bud,
                                            double d_bad, DiagPartial *out)
{
    for (int o = 16; o > 0; o >>= 1) {
        d_phi += __shfl_xor_sync(0xffffffffu, d_phi, o);
        d_E += __shfl_xor_sync(0xffffffffu, d_E, o);
        d_bud += __shfl_xor_sync(0xffffffffu, d_bud, o);
        d_u2 = fmax(d_u2, __shfl_xor_sync(0xffffffffu, d_u2, o));
        d_mumin = fmin(d_mumin, __shfl_xor_sync(0xffffffffu, d_mumin, o));
        d_mumax = fmax(d_mumax, __shfl_xor_sync(0xffffffffu, d_mumax, o));
        d_bad = fmax(d_bad, __shfl_xor_sync(0xffffffffu, d_bad, o));
    }
    constexpr int NW = NT / 32;
    __shared__ double red[7][NW];
    const int lane = tid & 31, wid = tid >> 5;
    if (lane == 0) {
        red[0][wid] = d_phi;
        red[1][wid] = d_E;
        red[2][wid] = d_u2;
        red[3][wid] = d_mumin;
        red[4][wid] = d_mumax;
        red[5][wid] = d_bud;
        red[6][wid] = d_bad;
    }
    __syncthreads();
    if (tid == 0) {
        DiagPartial o;
        o.sum_phi = 0.0, o.E = 0.0, o.u2max = 0.0, o.mu_min = DBL_MAX, o.mu_max = -DBL_MAX;
        o.budget = 0.0, o.nonfinite = 0.0, o.pad = 0.0;
        for (int w = 0; w < NW; ++w) {
            o.sum_phi += red[0][w];
            o.E += red[1][w];
            o.u2max = fmax(o.u2max, red[2][w]);
            o.mu_min = fmin(o.mu_min, red[3][w]);
            o.mu_max = fmax(o.mu_max, red[4][w]);
            o.budget += red[5][w];
            o.nonfinite = fmax(o.nonfinite, red[6][w]);
        }
        *out = o;
    }
}

// What bounds this pass: instruction issue and the latency of the pulls.
// Rebuilding 38 populations per node from their offsets took 1570 instructions
// per node with one node per thread (256^3 FP16: 1.135 ms, issue slots 60% busy
// at 16 warps per SM, DRAM 38%).  A thread owns two nodes adjacent in x
// instead: their arithmetic runs on the paired FP32 datapath (the same
// roundings in the same order), 16-bit values of a pair are loaded and stored
// as one 32-bit word where their alignment allows (every store, and the pulls
// without an x component), and the plane offsets of the asynchronous copies are
// formed once per march: 1030 instructions per node, 160^3 279 -> 233 us, whole
// 256^3 runs 1.40 -> 1.17 ms per step.  For rows of an even number of nodes, which is
// what those words need.  The asynchronous copies of phi and macros move pairs too
// (256^3 1068 -> 1061 us per step, 64^3 26.1 -> 25.2, 32^3 13.5 -> 12.4).
// Three CTAs of 128 threads per SM at 168 registers; four spill (83 ms against
// 47 ms per 40 steps at 256^3).  Measured and not kept, all bit-identical: the
// pulls staged a plane ahead in shared memory by 4-byte asynchronous copies
// (333 us: the load/store units take one word per thread at a time), the next
// plane's pulls in registers during the collisions at two CTAs per SM (238 us),
// or while its mu is formed (264 us: they spill).
template <class C, int PASS>
__global__ void __launch_bounds__(PAIR_NT, 3)
    d3q19_off_pass_kernel(const StepParams<float> P, PassArgs a, const OffBuf src, const OffBuf dst,
                          const float *__restrict__ target, const float *__restrict__ phif,
                          int planes)
{
    constexpr int PX = TX3 + 4, PY = TY3 + 4, PA = PX * PY;  // phi plane (halo 2)
    constexpr int MX = TX3 + 4, MY = TY3 + 2, MA = MX * MY;  // mu / macro plane (halo 1 used in
                                                             // x of the 2 stored: even pairs)
    constexpr int RP = 5, RM = 3;
    constexpr int MW = TX3 + 2, MN = MW * MY;  // nodes of a mu / macro plane
    __shared__ __align__(16) float phs[RP * PA];
    __shared__ __align__(16) float mus[RM * MA];
    // the source macros of the plane two ahead, copied while a plane is updated
    __shared__ __align__(16) float mraw[6 * MA];
    // per source node {alpha mu, A = 3p - 3/2 rho |u|^2, rho u_x, rho u_y, rho u_z, 9 / (2 rho)}:
    // g^eq_i = w_i (A + 3 c.j + (9/2)(c.j)^2 / rho); ring of three planes per quantity
    __shared__ __align__(16) float qs[6][RM * MA];

    const int bx = pdl_wait(blockIdx.x);
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const unsigned N = (unsigned)P.N;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TXP + tx;
    const int x0 = bx * TX3, y0 = blockIdx.y * TY3;
    const int z0 = blockIdx.z * planes, zend = min(z0 + planes, nz);
    const int x = x0 + 2 * tx, y = y0 + ty;
    const bool ok = x < nx && y < ny;  // (both nodes: nx is even)
    const unsigned plane = (unsigned)nx * ny;
    const float *ssc = after_wait(src.sc), *tsc = after_wait(target);
    const float s_f = __ldg(ssc), s_g = __ldg(ssc + 1);
    const float t_f = __ldg(tsc), t_g = __ldg(tsc + 1);
    const float it_f = 1.0f / t_f, it_g = 1.0f / t_g;  // powers of two: exact
    if ((PASS & PASS_STATE) && bx == 0 && blockIdx.y == 0 && blockIdx.z == 0 && tid == 0) {
        dst.sc[0] = t_f;
        dst.sc[1] = t_g;
    }

    // grids narrower than a tile plus halo wrap by division (uniform flags)
    const bool smx = nx < PX + 2, smy = ny < PY + 2, smz = nz < 8;
    // this thread's nodes of a mu / macro plane: ring index and in-plane offset in
    // the grid (nodes past the halo repeat)
    constexpr int KM = (MN + PAIR_NT - 1) / PAIR_NT;
    unsigned moff[KM];
    int mring[KM];  // index in a stored plane (row stride MX, x halo 2)
#pragma unroll
    for (int k = 0; k < KM; ++k) {
        const int q = tid + k * PAIR_NT;
        moff[k] = (unsigned)wrapc(y0 - 1 + q / MW, ny, smy) * nx + wrapc(x0 - 1 + q % MW, nx, smx);
        mring[k] = q / MW * MX + q % MW + 1;
    }
    // the pairs it copies of a phi plane and of a macro plane (a pair stays one
    // after the periodic wrap)
    constexpr int KP = (PA / 2 + PAIR_NT - 1) / PAIR_NT, KC = (MA / 2 + PAIR_NT - 1) / PAIR_NT;
    unsigned poff[KP], coff[KC];
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        const int q = 2 * (tid + k * PAIR_NT);
        poff[k] = (unsigned)wrapc(y0 - 2 + q / PX, ny, smy) * nx + wrapc(x0 - 2 + q % PX, nx, smx);
    }
#pragma unroll
    for (int k = 0; k < KC; ++k) {
        const int q = 2 * (tid + k * PAIR_NT);
        coff[k] = (unsigned)wrapc(y0 - 1 + q / MX, ny, smy) * nx + wrapc(x0 - 2 + q % MX, nx, smx);
    }
    // ring slots of plane z0 + d: phi (d + 2) mod 5, mu and macros (d + 1) mod 3
    auto wrapr = [](int v, int n) { return v >= n ? v - n : v; };
    // Eq. chemical_potencial with Eq. Laplace on D3Q19, from the phi slots of the
    // planes below, at and above into mu slot sm
    auto mu_plane = [&](int s_m, int s_0, int s_p, int sm) {
        const float *pm = phs + s_m * PA, *p0 = phs + s_0 * PA, *pp = phs + s_p * PA;
        float *d = mus + sm * MA;
#pragma unroll
        for (int k = 0; k < KM; ++k) {
            if (tid + k * PAIR_NT >= MN) break;
            const int c = mring[k] + PX;  // one phi row further (halo 2 against 1)
            const float v = p0[c];
            const float fa = (p0[c + 1] - v) + (p0[c - 1] - v) + (p0[c + PX] - v) +
                             (p0[c - PX] - v) + (pp[c] - v) + (pm[c] - v);
            const float ed = ((p0[c + PX + 1] - v) + (p0[c + PX - 1] - v) + (p0[c - PX + 1] - v) +
                              (p0[c - PX - 1] - v)) +
                             ((pp[c + 1] - v) + (pp[c - 1] - v) + (pm[c + 1] - v) + (pm[c - 1] - v)) +
                             ((pp[c + PX] - v) + (pp[c - PX] - v) + (pm[c + PX] - v) +
                              (pm[c - PX] - v));
            const float lap = (1.0f / 3.0f) * fa + (1.0f / 6.0f) * ed;
            d[mring[k]] = 4.0f * P.beta * (v - P.phil) * (v - P.phiv) * (v - P.phibar) - P.kappa * lap;
        }
    };
    // equilibrium data of the source state's macros (phi, mu, p, u) at ring index r of slot sm
    auto put_macros = [&](int sm, int r, const float m6[6]) {
        const float rho = P.rhov + (m6[0] - P.phiv) * P.drho;
        const int q = sm * MA + r;
        qs[0][q] = P.alpha * m6[1];
        qs[1][q] = 3.0f * m6[2] - 1.5f * rho * (m6[3] * m6[3] + m6[4] * m6[4] + m6[5] * m6[5]);
        qs[2][q] = rho * m6[3];
        qs[3][q] = rho * m6[4];
        qs[4][q] = rho * m6[5];
        qs[5][q] = 4.5f / rho;
    };

    double d_phi = 0.0, d_E = 0.0, d_u2 = 0.0, d_mumin = DBL_MAX, d_mumax = -DBL_MAX,
           d_bud = 0.0, d_bad = 0.0;

    for (int d = 0; d < 5; ++d) {
        const unsigned zo = (unsigned)wrapc(z0 - 2 + d, nz, smz) * plane;
#pragma unroll
        for (int k = 0; k < KP; ++k)
            if (2 * (tid + k * PAIR_NT) < PA)
                cp_async8(phs + d * PA + 2 * (tid + k * PAIR_NT), phif + (zo + poff[k]));
    }
    cp_commit();
    for (int d = 0; d < 3; ++d) {
        const unsigned zo = (unsigned)wrapc(z0 - 1 + d, nz, smz) * plane;
#pragma unroll
        for (int k = 0; k < KM; ++k) {
            if (tid + k * PAIR_NT >= MN) break;
            float m6[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) m6[c] = __ldg(src.M + (c * N + zo + moff[k]));
            put_macros(d, mring[k], m6);
        }
    }
    cp_wait_all();
    __syncthreads();
    for (int d = 0; d < 3; ++d) mu_plane(d, d + 1, d + 2, d);
    __syncthreads();

    // Plane zz + 3 of phi (into its ring slot) and the raw source macros of
    // plane zz + 2 (into mraw) are copied asynchronously while plane zz is
    // updated, so their loads overlap the node's own pulls and hold no
    // registers.  Ring use during the update of plane zz: phi zz-1..zz+1
    // (read) and zz+3 (being written); mu and macros zz-1..zz+1; once every
    // thread is past the update, macro plane zz+2 and mu plane zz+2 take the
    // slots of zz-1.
    const unsigned xw = ok ? (unsigned)x : 0, yw = ok ? (unsigned)y : 0;
    Nb b = make_nb((int)xw, (int)yw, z0, nx, ny, nz);
    const unsigned xp2 = (unsigned)wrap1((int)xw + 2, nx);  // the second node's +x neighbour
    int sp = 1, sq = 0;  // phi slot of plane zz - 1, mu / macro slot of plane zz - 1
    for (int zz = z0; zz < zend; ++zz) {
        const int sp0 = wrapr(sp + 1, RP), spp = wrapr(sp + 2, RP);
        const int sq0 = wrapr(sq + 1, RM), sqp = wrapr(sq + 2, RM);
        {
            const unsigned zo = (unsigned)wrapc(zz + 3, nz, smz) * plane;
            float *d = phs + wrapr(sp + 4, RP) * PA + 2 * tid;
#pragma unroll
            for (int k = 0; k < KP; ++k)
                if (2 * (tid + k * PAIR_NT) < PA) cp_async8(d + 2 * k * PAIR_NT, phif + (zo + poff[k]));
            const unsigned zm = (unsigned)wrapc(zz + 2, nz, smz) * plane;
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                if (2 * (tid + k * PAIR_NT) >= MA) break;
                const float *m = src.M + (zm + coff[k]);
#pragma unroll
                for (int c = 0; c < 6; ++c)
                    cp_async8(mraw + c * MA + 2 * (tid + k * PAIR_NT), m + (size_t)c * N);
            }
            cp_commit();
        }
        if (ok) {
        nb_plane(b, zz, nx, ny, nz);
        const unsigned row = b.zs[1] + b.ys[1], n = row + xw;
        // the offsets of the two nodes share one register (the first in the low half)
        unsigned hp[19], kp[19];
        auto pull = [&](const unsigned short *v, int i) -> unsigned {
            const unsigned r = i * N + b.zs[1 - c3z(i)] + b.ys[1 - c3y(i)];
            if (c3x(i) == 0) return __ldg(reinterpret_cast<const unsigned *>(v + (r + xw)));
            const unsigned ca = c3x(i) > 0 ? b.xs[0] : b.xs[2], cb = c3x(i) > 0 ? xw : xp2;
            return (unsigned)__ldg(v + (r + ca)) | ((unsigned)__ldg(v + (r + cb)) << 16);
        };
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            hp[i] = pull(src.h, i);
            kp[i] = pull(src.k, i);
        }
        // an FP32 value of each of the two nodes
        auto own = [&](const float *v) { return __ldg(reinterpret_cast<const float2 *>(v + n)); };
        float2 Sprev = f2(0.0f);
        if (PASS & (PASS_STATE | PASS_DIAG)) {
            Sprev = __ldcs(reinterpret_cast<const float2 *>(static_cast<const float *>(a.S) + n));
        }
        const float2 phi_hi = own(src.M), p_own = own(src.M + 2 * N);

        // populations after streaming, rebuilt from offsets and source macros
        const int c0 = (ty + 1) * MX + 2 * tx + 2;  // ring index of the first node (even)
        const float2 sf2 = f2(s_f), sg2 = f2(s_g);
        float2 fv[19], gv[19];
        float2 flo;  // rest population minus its high word phi_hi
        {
            const float2 ax = pair_at(qs[0] + sq0 * MA, c0, true);
            const float2 ay = pair_at(qs[1] + sq0 * MA, c0, true);
            flo = fma2(sf2, C::dec2(hp[0]), mul2(f2(-(2.0f / 3.0f)), ax));
            gv[0] = fma2(sg2, C::dec2(kp[0]),
                         fma2(f2(1.0f / 3.0f), ay, mul2(f2(-3.0f), p_own)));
        }
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const int sl = c3z(i) > 0 ? sq : (c3z(i) < 0 ? sqp : sq0);
            const int c = sl * MA + c0 - c3y(i) * MX - c3x(i);
            constexpr float w1 = (float)w3(1), w7 = (float)w3(7);
            const float2 w = f2(i <= 6 ? w1 : w7);
            const bool ev = c3x(i) == 0;
            fv[i] = fma2(w, pair_at(qs[0], c, ev), mul2(sf2, C::dec2(hp[i])));
            float2 jx = f2(0.0f), jy = f2(0.0f), jz = f2(0.0f);
            if (c3x(i)) jx = pair_at(qs[2], c, ev);
            if (c3y(i)) jy = pair_at(qs[3], c, ev);
            if (c3z(i)) jz = pair_at(qs[4], c, ev);
            const float2 cj = dot_c(c3x(i), c3y(i), c3z(i), jx, jy, jz);
            const float2 e = fma2(cj, fma2(pair_at(qs[5], c, ev), cj, f2(3.0f)),
                                  pair_at(qs[1], c, ev));
            gv[i] = fma2(sg2, C::dec2(kp[i]), mul2(w, e));
        }

        float2 snz = add2(fv[1], fv[2]), sg = add2(gv[1], gv[2]);
#pragma unroll
        for (int i = 3; i < 19; i += 2) {
            snz = add2(snz, add2(fv[i], fv[i + 1]));
            sg = add2(sg, add2(gv[i], gv[i + 1]));
        }
        // phi = phi_hi + (flo + snz) as an exact two-sum: phi (FP32) + r
        const float2 lo_sum = add2(flo, snz);
        const float2 phi = add2(phi_hi, lo_sum);
        const float2 bp = sub2(phi, phi_hi);
        const float2 r = add2(sub2(phi_hi, sub2(phi, bp)), sub2(lo_sum, bp));

        const int cp = (ty + 2) * PX + 2 * tx + 2;
        const float *m0 = mus + sq0 * MA, *mm = mus + sq * MA, *mp = mus + sqp * MA;
        const float2 mu = pair_at(m0, c0, true);
        float2 gp[3], gm[3];
        grad3_pair(phs + sp * PA, phs + sp0 * PA, phs + spp * PA, cp, PX, gp);
        grad3_pair(mm, m0, mp, c0, MX, gm);

        float2 F[3], gr[3], u[3];
        const float2 dphi = sub2(phi, f2(P.phiv));
        const float2 rho = fma2(dphi, f2(P.drho), f2(P.rhov));
        const float2 nu = fma2(dphi, f2(P.dnu), f2(P.nuv));
        const float2 inv_rho = make_float2(__fdividef(1.0f, rho.x), __fdividef(1.0f, rho.y));
        const float2 tg = fma2(f2(3.0f), nu, f2(0.5f));
        const float2 itg = make_float2(__fdividef(1.0f, tg.x), __fdividef(1.0f, tg.y));
        float2 j3[3] = {f2(0.0f), f2(0.0f), f2(0.0f)};
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            if (c3x(i)) j3[0] = c3x(i) > 0 ? add2(j3[0], gv[i]) : sub2(j3[0], gv[i]);
            if (c3y(i)) j3[1] = c3y(i) > 0 ? add2(j3[1], gv[i]) : sub2(j3[1], gv[i]);
            if (c3z(i)) j3[2] = c3z(i) > 0 ? add2(j3[2], gv[i]) : sub2(j3[2], gv[i]);
        }
        float2 ugr = f2(0.0f), uu = f2(0.0f), S = f2(0.0f);
        const float2 mphi = neg2(phi);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            F[d] = fma2(mphi, gm[d], f2(P.G[d]));
            gr[d] = mul2(f2(P.drho), gp[d]);
            u[d] = mul2(fma2(f2(0.5f), F[d], j3[d]), inv_rho);
            ugr = fma2(u[d], gr[d], ugr);
            uu = fma2(u[d], u[d], uu);
            S = fma2(u[d], gp[d], S);
        }
        const float2 p =
            mul2(f2(0.5f), fma2(mul2(f2(-0.5f), rho), uu, fma2(f2(0.5f), ugr, sg)));

        if (PASS & PASS_DIAG) {
            auto acc = [&](float ph, float rr, float rh, float u2f, float m, float Sn, float So,
                           float pp) {
                const double u2 = (double)u2f;
                d_phi += (double)ph + (double)rr;
                d_E += 0.5 * (double)rh * u2;
                d_u2 = fmax(d_u2, u2);
                d_mumin = fmin(d_mumin, (double)m);
                d_mumax = fmax(d_mumax, (double)m);
                d_bud += 1.5 * (double)Sn - 0.5 * (double)So;
                if (!isfinite(ph) || !isfinite(pp) || !isfinite(u2f) || !isfinite(m)) d_bad = 1.0;
            };
            acc(phi.x, r.x, rho.x, uu.x, mu.x, S.x, Sprev.x, p.x);
            acc(phi.y, r.y, rho.y, uu.y, mu.y, S.y, Sprev.y, p.y);
        }
        if (PASS & PASS_MACROS) {
            auto put = [&](double *o, double va, double vb) {
                o[n] = va;
                o[n + 1] = vb;
            };
            if (a.out_phi)
                put(a.out_phi, (double)phi.x + (double)r.x, (double)phi.y + (double)r.y);
            if (a.out_p) put(a.out_p, (double)p.x, (double)p.y);
            if (a.out_mu) put(a.out_mu, (double)mu.x, (double)mu.y);
            if (a.out_u) {
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    put(a.out_u + d * (size_t)N, (double)u[d].x, (double)u[d].y);
            }
        }
        if (PASS & PASS_STATE) {
            auto put = [&](float *o, float2 v) { __stcs(reinterpret_cast<float2 *>(o + n), v); };
            auto put16 = [&](unsigned short *o, float2 v) {
                __stcs(reinterpret_cast<unsigned *>(o + n), C::enc2(v));
            };
            put(static_cast<float *>(a.S), S);
            put(dst.M, phi);
            put(dst.M + N, mu);
            put(dst.M + 2 * N, p);
            put(dst.M + 3 * N, u[0]);
            put(dst.M + 4 * N, u[1]);
            put(dst.M + 5 * N, u[2]);
            {
                // B = phi + alpha sum_{i != 0} w_i (mu(x + c_i) - mu(x)) from the mu ring
                auto dm = [&](const float *pl, int o, bool ev) {
                    return sub2(pair_at(pl, c0 + o, ev), mu);
                };
                const float2 fa = add2(
                    add2(add2(add2(add2(dm(m0, 1, false), dm(m0, -1, false)), dm(m0, MX, true)),
                              dm(m0, -MX, true)),
                         dm(mp, 0, true)),
                    dm(mm, 0, true));
                const float2 e1 =
                    add2(add2(add2(dm(m0, MX + 1, false), dm(m0, MX - 1, false)),
                              dm(m0, -MX + 1, false)),
                         dm(m0, -MX - 1, false));
                const float2 e2 = add2(
                    add2(add2(dm(mp, 1, false), dm(mp, -1, false)), dm(mm, 1, false)),
                    dm(mm, -1, false));
                const float2 e3 = add2(
                    add2(add2(dm(mp, MX, true), dm(mp, -MX, true)), dm(mm, MX, true)),
                    dm(mm, -MX, true));
                const float2 ed = add2(add2(e1, e2), e3);
                put(dst.M + 6 * N,
                    fma2(f2(P.alpha), fma2(f2(1.0f / 18.0f), fa, mul2(f2(1.0f / 36.0f), ed)), phi));
            }
            // CH population (Eqs. BGK, F_i): offset = (f - f^eq)(1 - 1/tau_f) + F_i,
            // b = -5/2, -1, 1/2; the rest offset also carries the residual r of phi
            const float2 Sh = fma2(f2(1.5f), S, mul2(f2(-0.5f), Sprev));
            const float2 am = mul2(f2(P.alpha), mu);
            const float2 omf = f2(1.0f - P.inv_tauf), itf2 = f2(it_f), itg2 = f2(it_g);
            const float2 msnz = neg2(snz);
            const float2 d0 = fma2(f2(-(5.0f / 6.0f)), Sh,
                                   fma2(fma2(f2(2.0f / 3.0f), am, msnz), omf, r));
            put16(dst.h, mul2(d0, itf2));
            const float2 fa = mul2(f2(-(1.0f / 18.0f)), Sh), fe = mul2(f2(1.0f / 72.0f), Sh);
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                const float2 w = f2(-(float)w3(i));
                put16(dst.h + i * N,
                      mul2(fma2(fma2(w, am, fv[i]), omf, i <= 6 ? fa : fe), itf2));
            }
            // hydrodynamic population (Eqs. g_i, G_i): offset = (g - g^eq)(1 - 1/tau_g) + G_i
            const float2 kg = fma2(f2(-0.5f), itg, f2(1.0f)), omg = sub2(f2(1.0f), itg);
            const float2 p3 = mul2(f2(3.0f), p), mp3 = mul2(f2(-3.0f), p);
            const float2 A = fma2(mul2(f2(-1.5f), rho), uu, p3);
            put16(dst.k, mul2(mul2(sub2(gv[0], fma2(f2(1.0f / 3.0f), A, mp3)), omg), itg2));
            const float2 r45 = mul2(f2(4.5f), rho);
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                const int o = (i <= 6) ? (i % 2 ? i + 1 : i - 1)
                                       : (i <= 10 ? 17 - i : (i <= 14 ? 25 - i : 33 - i));
                if (o < i) continue;  // each pair once, from its first member
                const float wf = (float)w3(i);
                const float2 cu = dot_c(c3x(i), c3y(i), c3z(i), u[0], u[1], u[2]);
                const float2 cF = dot_c(c3x(i), c3y(i), c3z(i), F[0], F[1], F[2]);
                const float2 cg = dot_c(c3x(i), c3y(i), c3z(i), gr[0], gr[1], gr[2]);
                const float2 X = fma2(mul2(r45, cu), cu, A);           // eq_s = w X
                const float2 ra = mul2(f2(3.0f * wf), rho);            // eq_a = ra cu
                const float2 mra = mul2(f2(-3.0f * wf), rho);
                const float2 wk = mul2(f2(3.0f * wf), kg);             // G_a = wk cF
                const float2 mwk = mul2(f2(-3.0f * wf), kg);
                const float2 wkcu = mul2(wk, cu);                      // G_s = wk cu cg
                const float2 ti = fma2(mra, cu, fma2(f2(-wf), X, gv[i]));
                const float2 to = fma2(ra, cu, fma2(f2(-wf), X, gv[o]));
                put16(dst.k + i * N, mul2(fma2(wk, cF, fma2(wkcu, cg, mul2(ti, omg))), itg2));
                put16(dst.k + o * N, mul2(fma2(mwk, cF, fma2(wkcu, cg, mul2(to, omg))), itg2));
            }
        }
        }  // ok
        cp_wait_all();
        __syncthreads();
#pragma unroll
        for (int k = 0; k < KM; ++k) {
            if (tid + k * PAIR_NT >= MN) break;
            float m6[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) m6[c] = mraw[c * MA + mring[k]];
            put_macros(sq, mring[k], m6);
        }
        // phi planes zz + 1 .. zz + 3 -> mu plane zz + 2 in the slot of zz - 1
        mu_plane(spp, wrapr(sp + 3, RP), wrapr(sp + 4, RP), sq);
        __syncthreads();
        sp = sp0;
        sq = sq0;
    }

    if (PASS & PASS_DIAG)
        off_partial<PAIR_NT>(tid, d_phi, d_E, d_u2, d_mumin, d_mumax, d_bud, d_bad,
                             a.partials + (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + bx);
}

// The same pass with one node per thread, for rows of an odd number of nodes:
// there the two-node form has to load and store single values (twice the
// requests for the same sectors) and was 2 to 10% slower than this one
// (177 x 44 x 219 FP16 188 against 170 us per step).  Each value is formed by the same
// operations in the same order.  Which of them become multiply-adds is the
// compiler's choice here and written out above, after that choice: a test
// holds the two forms to the same bits.
template <class C, int PASS>
__global__ void __launch_bounds__(TX3 *TY3)
    d3q19_off_pass1_kernel(const StepParams<float> P, PassArgs a, const OffBuf src, const OffBuf dst,
                           const float *__restrict__ target, const float *__restrict__ phif,
                           int planes)
{
    constexpr int PX = TX3 + 4, PY = TY3 + 4, PA = PX * PY;  // phi plane (halo 2)
    constexpr int MX = TX3 + 2, MY = TY3 + 2, MA = MX * MY;  // mu / macro plane (halo 1)
    constexpr int RP = 5, RM = 3, RQ = 3;
    __shared__ float phs[RP * PA];
    __shared__ float mus[RM * MA];
    // the source macros of the plane two ahead, copied while a plane is updated
    __shared__ float mraw[6 * MA];
    // per source node: {alpha mu, A = 3p - 3/2 rho |u|^2, rho ux, rho uy} and
    // {rho uz, 9 / (2 rho)}: g^eq_i = w_i (A + 3 c.j + (9/2)(c.j)^2 / rho)
    __shared__ float4 qa[RQ * MA];
    __shared__ float2 qb[RQ * MA];

    const int bx = pdl_wait(blockIdx.x);
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const unsigned N = (unsigned)P.N;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX3 + tx;
    const int x0 = bx * TX3, y0 = blockIdx.y * TY3;
    const int z0 = blockIdx.z * planes, zend = min(z0 + planes, nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool col_ok = x < nx && y < ny;
    const unsigned plane = (unsigned)nx * ny;
    const float *ssc = after_wait(src.sc), *tsc = after_wait(target);
    const float s_f = __ldg(ssc), s_g = __ldg(ssc + 1);
    const float t_f = __ldg(tsc), t_g = __ldg(tsc + 1);
    const float it_f = 1.0f / t_f, it_g = 1.0f / t_g;  // powers of two: exact
    if ((PASS & PASS_STATE) && bx == 0 && blockIdx.y == 0 && blockIdx.z == 0 && tid == 0) {
        dst.sc[0] = t_f;
        dst.sc[1] = t_g;
    }

    auto pslot = [&](int zz) { return (zz - z0 + 2) % RP; };
    auto mslot = [&](int zz) { return (zz - z0 + 1) % RM; };
    auto qslot = [&](int zz) { return (zz - z0 + 1) % RQ; };

    // grids narrower than a tile plus halo wrap by division (uniform flags)
    const bool smx = nx < PX + 2, smy = ny < PY + 2, smz = nz < 8;
    auto load_phi_plane = [&](int zz) {
        float *d = phs + pslot(zz) * PA;
        const unsigned zo = (unsigned)wrapc(zz, nz, smz) * plane;
        for (int q = tid; q < PA; q += TX3 * TY3) {
            const int lx = q % PX, ly = q / PX;
            const unsigned xx = wrapc(x0 - 2 + lx, nx, smx), yy = wrapc(y0 - 2 + ly, ny, smy);
            d[q] = phif[zo + yy * nx + xx];
        }
    };
    // Eq. chemical_potencial with Eq. Laplace on D3Q19
    auto mu_plane = [&](int zz) {
        const float *pm = phs + pslot(zz - 1) * PA, *p0 = phs + pslot(zz) * PA,
                    *pp = phs + pslot(zz + 1) * PA;
        float *d = mus + mslot(zz) * MA;
        for (int q = tid; q < MA; q += TX3 * TY3) {
            const int lx = q % MX + 1, ly = q / MX + 1;
            const int c = ly * PX + lx;
            const float v = p0[c];
            const float fa = (p0[c + 1] - v) + (p0[c - 1] - v) + (p0[c + PX] - v) +
                             (p0[c - PX] - v) + (pp[c] - v) + (pm[c] - v);
            const float ed = ((p0[c + PX + 1] - v) + (p0[c + PX - 1] - v) + (p0[c - PX + 1] - v) +
                              (p0[c - PX - 1] - v)) +
                             ((pp[c + 1] - v) + (pp[c - 1] - v) + (pm[c + 1] - v) + (pm[c - 1] - v)) +
                             ((pp[c + PX] - v) + (pp[c - PX] - v) + (pm[c + PX] - v) +
                              (pm[c - PX] - v));
            const float lap = (1.0f / 3.0f) * fa + (1.0f / 6.0f) * ed;
            d[q] = 4.0f * P.beta * (v - P.phil) * (v - P.phiv) * (v - P.phibar) - P.kappa * lap;
        }
    };
    // equilibrium data of the source state's macros (ph, mu, p, u) at item q
    // of a macro plane (tile + 1 halo)
    auto put_macros = [&](int slot, int q, const float m6[6]) {
        const float rho = P.rhov + (m6[0] - P.phiv) * P.drho;
        qa[slot * MA + q] = make_float4(P.alpha * m6[1],
                                        3.0f * m6[2] - 1.5f * rho * (m6[3] * m6[3] + m6[4] * m6[4] + m6[5] * m6[5]),
                                        rho * m6[3], rho * m6[4]);
        qb[slot * MA + q] = make_float2(rho * m6[5], 4.5f / rho);
    };
    auto macro_node = [&](int zz, int q) {
        const unsigned m = (unsigned)wrapc(zz, nz, smz) * plane +
                           (unsigned)wrapc(y0 - 1 + q / MX, ny, smy) * nx + wrapc(x0 - 1 + q % MX, nx, smx);
        return m;
    };
    auto macro_plane = [&](int zz) {
        for (int q = tid; q < MA; q += TX3 * TY3) {
            const unsigned m = macro_node(zz, q);
            float m6[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) m6[k] = __ldg(src.M + k * N + m);
            put_macros(qslot(zz), q, m6);
        }
    };
    auto grad3 = [&](const float *m, const float *c0, const float *p, int c, int SX, float out[3]) {
        out[0] = (1.0f / 6.0f) * (c0[c + 1] - c0[c - 1]) +
                 (1.0f / 12.0f) * ((c0[c + SX + 1] - c0[c + SX - 1]) + (c0[c - SX + 1] - c0[c - SX - 1]) +
                                   (p[c + 1] - p[c - 1]) + (m[c + 1] - m[c - 1]));
        out[1] = (1.0f / 6.0f) * (c0[c + SX] - c0[c - SX]) +
                 (1.0f / 12.0f) * ((c0[c + SX + 1] - c0[c - SX + 1]) + (c0[c + SX - 1] - c0[c - SX - 1]) +
                                   (p[c + SX] - p[c - SX]) + (m[c + SX] - m[c - SX]));
        out[2] = (1.0f / 6.0f) * (p[c] - m[c]) +
                 (1.0f / 12.0f) * ((p[c + 1] - m[c + 1]) + (p[c - 1] - m[c - 1]) +
                                   (p[c + SX] - m[c + SX]) + (p[c - SX] - m[c - SX]));
    };

    double d_phi = 0.0, d_E = 0.0, d_u2 = 0.0, d_mumin = DBL_MAX, d_mumax = -DBL_MAX,
           d_bud = 0.0, d_bad = 0.0;

    for (int q = 0; q < 5; ++q) load_phi_plane(z0 - 2 + q);
    macro_plane(z0 - 1);
    macro_plane(z0);
    macro_plane(z0 + 1);
    __syncthreads();
    mu_plane(z0 - 1);
    mu_plane(z0);
    mu_plane(z0 + 1);
    __syncthreads();

    // Plane zz + 3 of phi (into its ring slot) and the raw source macros of
    // plane zz + 2 (into mraw) are copied asynchronously while plane zz is
    // updated, so their loads overlap the node's own pulls and hold no
    // registers.  Ring use during the update of plane zz: phi zz-1..zz+1
    // (read) and zz+3 (being written); mu and macros zz-1..zz+1; once every
    // thread is past the update, macro plane zz+2 and mu plane zz+2 take the
    // slots of zz-1.
    const unsigned xw = col_ok ? (unsigned)x : 0, yw = col_ok ? (unsigned)y : 0;
    Nb b = make_nb(xw, yw, z0, nx, ny, nz);
    for (int zz = z0; zz < zend; ++zz) {
        {
            const unsigned zo = (unsigned)wrapc(zz + 3, nz, smz) * plane;
            float *d = phs + pslot(zz + 3) * PA;
            for (int q = tid; q < PA; q += TX3 * TY3) {
                const unsigned xx = wrapc(x0 - 2 + q % PX, nx, smx), yy = wrapc(y0 - 2 + q / PX, ny, smy);
                cp_async4(d + q, phif + (zo + yy * nx + xx));
            }
            for (int q = tid; q < MA; q += TX3 * TY3) {
                const unsigned m = macro_node(zz + 2, q);
#pragma unroll
                for (int c = 0; c < 6; ++c) cp_async4(mraw + c * MA + q, src.M + ((size_t)c * N + m));
            }
            cp_commit();
        }
        if (col_ok) {
        nb_plane(b, zz, nx, ny, nz);
        const unsigned n = b.at(0, 0, 0);
        // the two 16-bit offsets of direction i share one register
        unsigned hk[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const unsigned s = b.at(-c3x(i), -c3y(i), -c3z(i));
            hk[i] = (unsigned)__ldg(src.h + (i * N + s)) | ((unsigned)__ldg(src.k + (i * N + s)) << 16);
        }
        auto hr = [&](int i) { return (unsigned short)(hk[i] & 0xffffu); };
        auto kr = [&](int i) { return (unsigned short)(hk[i] >> 16); };
        float Sprev = 0.0f;
        if (PASS & (PASS_STATE | PASS_DIAG)) Sprev = __ldcs(static_cast<const float *>(a.S) + n);
        const float phi_hi = __ldg(src.M + n), p_own = __ldg(src.M + 2 * N + n);

        // populations after streaming, rebuilt from offsets and source macros
        const int cq = (ty + 1) * MX + (tx + 1);
        float fv[19], gv[19];
        float flo;  // rest population minus its high word phi_hi
        {
            const float4 A0 = qa[qslot(zz) * MA + cq];
            flo = -(2.0f / 3.0f) * A0.x + s_f * C::dec(hr(0));
            gv[0] = (1.0f / 3.0f) * A0.y - 3.0f * p_own + s_g * C::dec(kr(0));
        }
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const int c = qslot(zz - c3z(i)) * MA + cq - c3y(i) * MX - c3x(i);
            const float4 A = qa[c];
            const float2 B = qb[c];
            const float w = (float)w3(i);
            fv[i] = w * A.x + s_f * C::dec(hr(i));
            float cj = 0.0f;
            if (c3x(i)) cj += (float)c3x(i) * A.z;
            if (c3y(i)) cj += (float)c3y(i) * A.w;
            if (c3z(i)) cj += (float)c3z(i) * B.x;
            gv[i] = w * (A.y + cj * (3.0f + B.y * cj)) + s_g * C::dec(kr(i));
        }

        float snz = 0.0f, sg = 0.0f;
#pragma unroll
        for (int i = 1; i < 19; i += 2) {
            snz += fv[i] + fv[i + 1];
            sg += gv[i] + gv[i + 1];
        }
        // phi = phi_hi + (flo + snz) as an exact two-sum: phi (FP32) + r
        const float lo_sum = flo + snz;
        const float phi = phi_hi + lo_sum;
        const float bp = phi - phi_hi;
        const float r = (phi_hi - (phi - bp)) + (lo_sum - bp);

        const int cp = (ty + 2) * PX + (tx + 2), cm = cq;
        const float *mz = mus + mslot(zz) * MA;
        const float mu = mz[cm];
        float gp[3], gm[3];
        grad3(phs + pslot(zz - 1) * PA, phs + pslot(zz) * PA, phs + pslot(zz + 1) * PA, cp, PX, gp);
        grad3(mus + mslot(zz - 1) * MA, mz, mus + mslot(zz + 1) * MA, cm, MX, gm);

        float F[3], gr[3], u[3];
        const float dphi = phi - P.phiv;
        const float rho = P.rhov + dphi * P.drho;
        const float nu = P.nuv + dphi * P.dnu;
        const float inv_rho = __fdividef(1.0f, rho);
        const float itg = __fdividef(1.0f, 0.5f + 3.0f * nu);
        float j3[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            if (c3x(i)) j3[0] += (float)c3x(i) * gv[i];
            if (c3y(i)) j3[1] += (float)c3y(i) * gv[i];
            if (c3z(i)) j3[2] += (float)c3z(i) * gv[i];
        }
        float ugr = 0.0f, uu = 0.0f, S = 0.0f;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            F[d] = -phi * gm[d] + P.G[d];
            gr[d] = P.drho * gp[d];
            u[d] = (j3[d] + 0.5f * F[d]) * inv_rho;
            ugr += u[d] * gr[d];
            uu += u[d] * u[d];
            S += u[d] * gp[d];
        }
        const float p = 0.5f * (sg + 0.5f * ugr - 0.5f * rho * uu);

        if (PASS & PASS_DIAG) {
            const double u2 = (double)uu;
            d_phi += (double)phi + (double)r;
            d_E += 0.5 * (double)rho * u2;
            d_u2 = fmax(d_u2, u2);
            d_mumin = fmin(d_mumin, (double)mu);
            d_mumax = fmax(d_mumax, (double)mu);
            d_bud += 1.5 * (double)S - 0.5 * (double)Sprev;
            if (!isfinite(phi) || !isfinite(p) || !isfinite(uu) || !isfinite(mu)) d_bad = 1.0;
        }
        if (PASS & PASS_MACROS) {
            if (a.out_phi) a.out_phi[n] = (double)phi + (double)r;
            if (a.out_p) a.out_p[n] = (double)p;
            if (a.out_mu) a.out_mu[n] = (double)mu;
            if (a.out_u) {
                a.out_u[n] = (double)u[0];
                a.out_u[(size_t)N + n] = (double)u[1];
                a.out_u[2 * (size_t)N + n] = (double)u[2];
            }
        }
        if (PASS & PASS_STATE) {
            __stcs(static_cast<float *>(a.S) + n, S);
            __stcs(dst.M + n, phi);
            __stcs(dst.M + N + n, mu);
            __stcs(dst.M + 2 * N + n, p);
            __stcs(dst.M + 3 * N + n, u[0]);
            __stcs(dst.M + 4 * N + n, u[1]);
            __stcs(dst.M + 5 * N + n, u[2]);
            {
                // B = phi + alpha sum_{i != 0} w_i (mu(x + c_i) - mu(x)) from the mu ring
                const float *m0 = mz, *mm = mus + mslot(zz - 1) * MA, *mp = mus + mslot(zz + 1) * MA;
                const float fa = (m0[cm + 1] - mu) + (m0[cm - 1] - mu) + (m0[cm + MX] - mu) +
                                 (m0[cm - MX] - mu) + (mp[cm] - mu) + (mm[cm] - mu);
                const float ed = ((m0[cm + MX + 1] - mu) + (m0[cm + MX - 1] - mu) +
                                  (m0[cm - MX + 1] - mu) + (m0[cm - MX - 1] - mu)) +
                                 ((mp[cm + 1] - mu) + (mp[cm - 1] - mu) + (mm[cm + 1] - mu) +
                                  (mm[cm - 1] - mu)) +
                                 ((mp[cm + MX] - mu) + (mp[cm - MX] - mu) + (mm[cm + MX] - mu) +
                                  (mm[cm - MX] - mu));
                __stcs(dst.M + 6 * N + n, phi + P.alpha * ((1.0f / 18.0f) * fa + (1.0f / 36.0f) * ed));
            }
            // CH population (Eqs. BGK, F_i): offset = (f - f^eq)(1 - 1/tau_f) + F_i,
            // b = -5/2, -1, 1/2; the rest offset also carries the residual r of phi
            const float Sh = 1.5f * S - 0.5f * Sprev;
            const float am = P.alpha * mu;
            const float omf = 1.0f - P.inv_tauf;
            const float d0 = ((2.0f / 3.0f) * am - snz) * omf + r - (5.0f / 6.0f) * Sh;
            __stcs(dst.h + n, C::enc(d0 * it_f));
            const float fa = -(1.0f / 18.0f) * Sh, fe = (1.0f / 72.0f) * Sh;
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                const float w = (float)w3(i);
                __stcs(dst.h + (i * N + n), C::enc(((fv[i] - w * am) * omf + (i <= 6 ? fa : fe)) * it_f));
            }
            // hydrodynamic population (Eqs. g_i, G_i): offset = (g - g^eq)(1 - 1/tau_g) + G_i
            const float kg = 1.0f - 0.5f * itg, omg = 1.0f - itg;
            const float A = 3.0f * p - 1.5f * rho * uu;
            __stcs(dst.k + n, C::enc((gv[0] - ((1.0f / 3.0f) * A - 3.0f * p)) * omg * it_g));
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                const int o = (i <= 6) ? (i % 2 ? i + 1 : i - 1)
                                       : (i <= 10 ? 17 - i : (i <= 14 ? 25 - i : 33 - i));
                if (o < i) continue;  // each pair once, from its first member
                const float w = (float)w3(i);
                const float cu = (float)c3x(i) * u[0] + (float)c3y(i) * u[1] + (float)c3z(i) * u[2];
                const float cF = (float)c3x(i) * F[0] + (float)c3y(i) * F[1] + (float)c3z(i) * F[2];
                const float cg = (float)c3x(i) * gr[0] + (float)c3y(i) * gr[1] + (float)c3z(i) * gr[2];
                const float eq_s = w * (A + 4.5f * rho * cu * cu), eq_a = 3.0f * w * rho * cu;
                const float G_s = 3.0f * w * kg * cu * cg, G_a = 3.0f * w * kg * cF;
                __stcs(dst.k + (i * N + n), C::enc(((gv[i] - eq_s - eq_a) * omg + G_s + G_a) * it_g));
                __stcs(dst.k + (o * N + n), C::enc(((gv[o] - eq_s + eq_a) * omg + G_s - G_a) * it_g));
            }
        }
        }  // col_ok
        cp_wait_all();
        __syncthreads();
        for (int q = tid; q < MA; q += TX3 * TY3) {  // own copies: no barrier needed
            float m6[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) m6[c] = mraw[c * MA + q];
            put_macros(qslot(zz + 2), q, m6);
        }
        mu_plane(zz + 2);
        __syncthreads();
    }

    if (PASS & PASS_DIAG)
        off_partial<TX3 * TY3>(tid, d_phi, d_E, d_u2, d_mumin, d_mumax, d_bud, d_bad,
                               a.partials + (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + bx);
}

// ------------------------------------------------- state in the paper's form

// equilibria of the stored macros of node m (the arithmetic of the pass kernel)
struct EqData {
    float q0, A, j[3], q5;
};
__device__ inline EqData eq_data(const StepParams<float> &P, const float *M, size_t N, size_t m)
{
    const float ph = M[m], mu = M[N + m], p = M[2 * N + m];
    const float u[3] = {M[3 * N + m], M[4 * N + m], M[5 * N + m]};
    const float rho = P.rhov + (ph - P.phiv) * P.drho;
    EqData e;
    e.q0 = P.alpha * mu;
    e.A = 3.0f * p - 1.5f * rho * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    for (int d = 0; d < 3; ++d) e.j[d] = rho * u[d];
    e.q5 = 4.5f / rho;
    return e;
}
__device__ inline double feq_of(const EqData &e, float phi_hi, int i)
{
    return i == 0 ? (double)phi_hi - (double)((2.0f / 3.0f) * e.q0) : (double)((float)w3(i) * e.q0);
}
__device__ inline double geq_of(const EqData &e, float p, int i)
{
    if (i == 0) return (double)((1.0f / 3.0f) * e.A - 3.0f * p);
    float cj = 0.0f;
    if (c3x(i)) cj += (float)c3x(i) * e.j[0];
    if (c3y(i)) cj += (float)c3y(i) * e.j[1];
    if (c3z(i)) cj += (float)c3z(i) * e.j[2];
    return (double)((float)w3(i) * (e.A + cj * (3.0f + e.q5 * cj)));
}

// Initial state: macros (phi0, mu0, p = 0, u = 0) at every node, f_i(x, 0) =
// f^eq_i(phi0(x), mu0(x)) stored at x - c_i as an offset from the equilibrium
// of the storing node's macros; g = g^eq (offsets 0).  Two passes: the first
// forms mu0 and the node's moving values, fa on the faces (FP64 scratch) and
// exactly half of it on the edges, the second stores their differences from the
// neighbours' equilibria.  Of the state only the parity that is initialised is
// written: phi0 may lie in the other one.  The FP64 pipe bounds both; the scales
// are powers of two, so the values are taken times 1/s_f before their differences
// are formed, which is exact and rounds to FP32 and to storage as the divided
// difference does, down to its smallest values, and takes one FP64 operation (a
// divide of its own for each of the 19 values made this 13.1 ms at 256^3, against
// 3.0 ms now).
template <class C>
__global__ void __launch_bounds__(256)
    d3q19_off_init_macros_k(const StepParams<double> Pd, const StepParams<float> P,
                            const double *__restrict__ phi0, double *__restrict__ fa, OffBuf o,
                            float *__restrict__ S, float s_f, float s_g, double inv)
{
    const unsigned N = (unsigned)P.N, n = blockIdx.x * 256u + threadIdx.x;
    if (n == 0) {
        o.sc[0] = s_f;
        o.sc[1] = s_g;
    }
    if (n >= N) return;
    const unsigned nx = P.nx, ny = P.ny;
    const unsigned r = n / nx;
    const Nb b = make_nb((int)(n - r * nx), (int)(r % ny), (int)(r / ny), P.nx, P.ny, P.nz);
    const double c = __ldg(phi0 + n);
    const double mu = mu_of_field(Pd, phi0, b, c), am = Pd.alpha * mu;
    static_assert(2.0 * w3(7) == w3(1), "edge values are half the face values");
    fa[n] = (inv * w3(1)) * am;
    const float phi_hi = (float)c, mu_f = (float)mu;
    o.M[n] = phi_hi;
    o.M[N + n] = mu_f;
#pragma unroll
    for (int k = 2; k < 6; ++k) o.M[k * N + n] = 0.0f;
    S[n] = 0.0f;
    const float q0 = P.alpha * mu_f;
    const double eq = (double)phi_hi - (double)((2.0f / 3.0f) * q0);
    o.h[n] = C::enc((float)(inv * (c - (1.0 - w3(0)) * am - eq)));
}

template <class C>
__global__ void __launch_bounds__(256)
    d3q19_off_init_k(const StepParams<float> P, const double *__restrict__ fa, OffBuf o, float inv)
{
    const unsigned N = (unsigned)P.N, n = blockIdx.x * 256u + threadIdx.x;
    if (n >= N) return;
    const unsigned nx = P.nx, ny = P.ny;
    const unsigned r = n / nx;
    const Nb b = make_nb((int)(n - r * nx), (int)(r % ny), (int)(r / ny), P.nx, P.ny, P.nz);
    const float q0 = P.alpha * o.M[N + n];
    const double eqa = (double)((float)w3(1) * q0 * inv), eqe = (double)((float)w3(7) * q0 * inv);
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const unsigned m = b.at(c3x(i), c3y(i), c3z(i));
        const double d = i <= 6 ? __ldg(fa + m) - eqa : fma(0.5, __ldg(fa + m), -eqe);
        o.h[i * N + n] = C::enc((float)d);
    }
#pragma unroll
    for (int i = 0; i < 19; ++i) o.k[i * N + n] = 0;  // +0 in both formats
}

template <class C>
__global__ void d3q19_off_get_k(const StepParams<float> P, const OffBuf o,
                                const float *__restrict__ S, double *fo, double *go, double *So)
{
    const size_t N = (size_t)P.N;
    const size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x = (int)(n % nx), y = (int)((n / nx) % ny), z = (int)(n / ((size_t)nx * ny));
    const Nb b = make_nb(x, y, z, nx, ny, nz);
    const double s_f = o.sc[0], s_g = o.sc[1];
    for (int i = 0; i < 19; ++i) {
        const unsigned m = b.at(-c3x(i), -c3y(i), -c3z(i));
        const EqData e = eq_data(P, o.M, N, m);
        if (fo) fo[i * N + n] = feq_of(e, o.M[m], i) + s_f * (double)C::dec(o.h[i * N + m]);
        if (go) go[i * N + n] = geq_of(e, o.M[2 * N + m], i) + s_g * (double)C::dec(o.k[i * N + m]);
    }
    if (So) So[n] = (double)S[n];
}

// macros of the storing node from its own stored values: phi = sum f*,
// mu from sum_{i != 0} f* = (1 - w0) alpha mu, u = sum c g* / rho,
// p = sum_{i != 0} g* / 2; the offsets carry the rest exactly (up to rounding)
template <class C>
__global__ void d3q19_off_set_k(const StepParams<float> P, OffBuf o, float *__restrict__ S,
                                const double *fi, const double *gi, const double *Si, float s_f,
                                float s_g)
{
    const size_t N = (size_t)P.N;
    const size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n == 0) {
        o.sc[0] = s_f;
        o.sc[1] = s_g;
    }
    if (n >= N) return;
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x = (int)(n % nx), y = (int)((n / nx) % ny), z = (int)(n / ((size_t)nx * ny));
    const Nb b = make_nb(x, y, z, nx, ny, nz);
    double fs[19], gs[19];
    double sphi = 0.0, snz = 0.0, sg = 0.0, j[3] = {0.0, 0.0, 0.0};
    for (int i = 0; i < 19; ++i) {
        const unsigned m = b.at(c3x(i), c3y(i), c3z(i));
        fs[i] = fi[i * N + m];
        gs[i] = gi[i * N + m];
        sphi += fs[i];
        if (i) {
            snz += fs[i];
            sg += gs[i];
            j[0] += c3x(i) * gs[i];
            j[1] += c3y(i) * gs[i];
            j[2] += c3z(i) * gs[i];
        }
    }
    const float phi_hi = (float)sphi;
    const float rho = P.rhov + (phi_hi - P.phiv) * P.drho;
    o.M[n] = phi_hi;
    o.M[N + n] = (float)(snz / ((1.0 - w3(0)) * (double)P.alpha));
    o.M[2 * N + n] = (float)(0.5 * sg);
    for (int d = 0; d < 3; ++d) o.M[(3 + d) * N + n] = (float)(j[d] / (double)rho);
    S[n] = (float)Si[n];
    const EqData e = eq_data(P, o.M, N, n);
    for (int i = 0; i < 19; ++i) {
        o.h[i * N + n] = C::enc((float)((fs[i] - feq_of(e, phi_hi, i)) / (double)s_f));
        o.k[i * N + n] = C::enc((float)((gs[i] - geq_of(e, o.M[2 * N + n], i)) / (double)s_g));
    }
}

// one population value of the paper's form written into the storage
template <class C>
__global__ void d3q19_off_poke_k(const StepParams<float> P, OffBuf o, int field, int i,
                                 size_t m, double value)
{
    const size_t N = (size_t)P.N;
    const EqData e = eq_data(P, o.M, N, m);
    if (field == 0)
        o.h[i * N + m] = C::enc((float)((value - feq_of(e, o.M[m], i)) / (double)o.sc[0]));
    else
        o.k[i * N + m] = C::enc((float)((value - geq_of(e, o.M[2 * N + m], i)) / (double)o.sc[1]));
}

// ---------------------------------------------------------------- scales

// max over |stored value| bit patterns (monotonic in the magnitude for both
// formats; NaN patterns are larger than INF_BITS) of the f and the g offsets
// (blockIdx.y 0, 1) into out[0], out[1].  HBM bounds it: eight values per
// 16-byte load, four loads in flight per thread (one value at a time took
// 885 us per field at 256^3, 0.7 TB/s).  v is 16-byte aligned.
__global__ void __launch_bounds__(256)
    off_absmax_k(const unsigned short *__restrict__ f, const unsigned short *__restrict__ g,
                 size_t count, unsigned *__restrict__ out)
{
    const unsigned short *v = blockIdx.y ? g : f;
    const uint4 *w = reinterpret_cast<const uint4 *>(v);
    const size_t nv = count / 8, step = (size_t)gridDim.x * 256;
    const size_t i0 = (size_t)blockIdx.x * 256 + threadIdx.x;
    unsigned m2 = 0;  // two 16-bit maxima
    auto take = [&](uint4 q) {
        m2 = __vmaxu2(m2, q.x & 0x7fff7fffu);
        m2 = __vmaxu2(m2, q.y & 0x7fff7fffu);
        m2 = __vmaxu2(m2, q.z & 0x7fff7fffu);
        m2 = __vmaxu2(m2, q.w & 0x7fff7fffu);
    };
    size_t i = i0;
    for (; i + 3 * step < nv; i += 4 * step) {
        const uint4 a = __ldg(w + i), b = __ldg(w + i + step), c = __ldg(w + i + 2 * step),
                    d = __ldg(w + i + 3 * step);
        take(a);
        take(b);
        take(c);
        take(d);
    }
    for (; i < nv; i += step) take(__ldg(w + i));
    unsigned m = max(m2 & 0xffffu, m2 >> 16);
    if (i0 < count - nv * 8) m = max(m, (unsigned)(__ldg(v + nv * 8 + i0) & 0x7fffu));
    m = __reduce_max_sync(0xffffffffu, m);
    __shared__ unsigned wm[8];
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) m = max(m, wm[k]);
        if (m) atomicMax(out + blockIdx.y, m);
    }
}

template <class C>
__global__ void off_target_k(const OffBuf cur, const unsigned *__restrict__ maxbits,
                             float *__restrict__ target)
{
    for (int k = 0; k < 2; ++k) {
        const unsigned bits = maxbits[k];
        if (bits >= C::INF_BITS) continue;  // overflowed or NaN: keep (diagnostics report it)
        const float m = C::dec((unsigned short)bits) * cur.sc[k];
        float t = OFFSET_SCALE_FLOOR;
        if (m > 0.0f) {
            int e;
            frexpf(m * (1.0f / OFFSET_HEADROOM), &e);
            t = fmaxf(t, ldexpf(1.0f, e));
        }
        target[k] = t;
    }
}

template <class C>
int off_ctas_per_sm_t(bool even)
{
    int n = 0;
    cudaError_t e = even ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                               &n, d3q19_off_pass_kernel<C, PASS_STATE>, PAIR_NT, 0)
                         : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                               &n, d3q19_off_pass1_kernel<C, PASS_STATE>, TX3 * TY3, 0);
    return e == cudaSuccess && n > 0 ? n : 2;
}

template <class C, int PASS>
cudaError_t launch_off(const StepParams<float> &P, const PassArgs &a, const LaunchShape &s,
                       float *phi, const float *target, cudaStream_t st)
{
    const OffBuf src = off_view(a.f_src, a.g_src, P.N), dst = off_view(a.f_dst, a.g_dst, P.N);
    const dim3 pg((P.nx + PHI_TX - 1) / PHI_TX, P.ny, P.nz);
    const cudaError_t e = launch_pdl(d3q19_off_phi_kernel<C>, pg, PHI_TX, 0, st, P, src, phi);
    if (e != cudaSuccess) return e;
    const dim3 grid(s.grid_x, s.grid_y, s.nblocks / (s.grid_x * s.grid_y));
    if (P.nx % 2 == 0)
        return launch_pdl(d3q19_off_pass_kernel<C, PASS>, grid, dim3(TXP, TY3), 0, st, P, a, src,
                          dst, target, phi, s.rows);
    return launch_pdl(d3q19_off_pass1_kernel<C, PASS>, grid, dim3(TX3, TY3), 0, st, P, a, src, dst,
                      target, phi, s.rows);
}

template <class C>
cudaError_t pass_off_t(int pass, const StepParams<float> &P, const PassArgs &a,
                       const LaunchShape &s, float *phi, const float *target, cudaStream_t st)
{
    switch (pass) {
    case PASS_STATE: return launch_off<C, PASS_STATE>(P, a, s, phi, target, st);
    case PASS_STATE | PASS_DIAG: return launch_off<C, PASS_STATE | PASS_DIAG>(P, a, s, phi, target, st);
    case PASS_MACROS: return launch_off<C, PASS_MACROS>(P, a, s, phi, target, st);
    case PASS_DIAG: return launch_off<C, PASS_DIAG>(P, a, s, phi, target, st);
    case PASS_MACROS | PASS_DIAG: return launch_off<C, PASS_MACROS | PASS_DIAG>(P, a, s, phi, target, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int d3q19_off_ctas_per_sm(int codec, int nx)
{
    const bool even = nx % 2 == 0;
    return codec == OFFSET_F16 ? off_ctas_per_sm_t<CodecF16>(even) : off_ctas_per_sm_t<CodecBF16>(even);
}

cudaError_t d3q19_off_pass(int codec, int pass, const void *params32, const PassArgs &a,
                           const LaunchShape &s, void *phi_work, const float *target,
                           cudaStream_t st)
{
    const StepParams<float> &P = *static_cast<const StepParams<float> *>(params32);
    return codec == OFFSET_F16
               ? pass_off_t<CodecF16>(pass, P, a, s, (float *)phi_work, target, st)
               : pass_off_t<CodecBF16>(pass, P, a, s, (float *)phi_work, target, st);
}

cudaError_t d3q19_off_init(int codec, const void *params64, const void *params32,
                           const double *phi0, double *tmp, void *f, void *g, void *S,
                           const float *target_host, cudaStream_t st)
{
    const StepParams<double> &Pd = *static_cast<const StepParams<double> *>(params64);
    const StepParams<float> &P = *static_cast<const StepParams<float> *>(params32);
    const unsigned nb = (unsigned)((P.N + 255) / 256);
    const OffBuf o = off_view(f, g, P.N);
    const float sf = target_host[0], sg = target_host[1];
    const double inv = 1.0 / sf;
    if (codec == OFFSET_F16) {
        d3q19_off_init_macros_k<CodecF16><<<nb, 256, 0, st>>>(Pd, P, phi0, tmp, o, (float *)S, sf,
                                                              sg, inv);
        d3q19_off_init_k<CodecF16><<<nb, 256, 0, st>>>(P, tmp, o, (float)inv);
    } else {
        d3q19_off_init_macros_k<CodecBF16><<<nb, 256, 0, st>>>(Pd, P, phi0, tmp, o, (float *)S, sf,
                                                               sg, inv);
        d3q19_off_init_k<CodecBF16><<<nb, 256, 0, st>>>(P, tmp, o, (float)inv);
    }
    d3q19_off_prep_k<<<dim3((P.nx + PHI_TX - 1) / PHI_TX, P.ny, P.nz), PHI_TX, 0, st>>>(P, o);
    return cudaGetLastError();
}

cudaError_t d3q19_off_get_state(int codec, const void *params32, const void *f, const void *g,
                                const void *S, double *fo, double *go, double *So, cudaStream_t st)
{
    const StepParams<float> &P = *static_cast<const StepParams<float> *>(params32);
    const unsigned nb = (unsigned)((P.N + 255) / 256);
    const OffBuf o = off_view(f, g, P.N);
    if (codec == OFFSET_F16)
        d3q19_off_get_k<CodecF16><<<nb, 256, 0, st>>>(P, o, (const float *)S, fo, go, So);
    else
        d3q19_off_get_k<CodecBF16><<<nb, 256, 0, st>>>(P, o, (const float *)S, fo, go, So);
    return cudaGetLastError();
}

cudaError_t d3q19_off_set_state(int codec, const void *params32, void *f, void *g, void *S,
                                const double *fi, const double *gi, const double *Si,
                                const float *target_host, cudaStream_t st)
{
    const StepParams<float> &P = *static_cast<const StepParams<float> *>(params32);
    const unsigned nb = (unsigned)((P.N + 255) / 256);
    const OffBuf o = off_view(f, g, P.N);
    if (codec == OFFSET_F16)
        d3q19_off_set_k<CodecF16><<<nb, 256, 0, st>>>(P, o, (float *)S, fi, gi, Si,
                                                      target_host[0], target_host[1]);
    else
        d3q19_off_set_k<CodecBF16><<<nb, 256, 0, st>>>(P, o, (float *)S, fi, gi, Si,
                                                       target_host[0], target_host[1]);
    d3q19_off_prep_k<<<dim3((P.nx + PHI_TX - 1) / PHI_TX, P.ny, P.nz), PHI_TX, 0, st>>>(P, o);
    return cudaGetLastError();
}

cudaError_t d3q19_off_poke(int codec, const void *params32, void *f, void *g, int field, int i,
                           size_t m, double value, cudaStream_t st)
{
    const StepParams<float> &P = *static_cast<const StepParams<float> *>(params32);
    const OffBuf o = off_view(f, g, P.N);
    if (codec == OFFSET_F16)
        d3q19_off_poke_k<CodecF16><<<1, 1, 0, st>>>(P, o, field, i, m, value);
    else
        d3q19_off_poke_k<CodecBF16><<<1, 1, 0, st>>>(P, o, field, i, m, value);
    return cudaGetLastError();
}

cudaError_t offset_refresh(int codec, long long N, int Q, const void *f, const void *g,
                           unsigned *maxbits, float *target, int num_sms, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(maxbits, 0, 2 * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    const size_t count = (size_t)Q * (size_t)N;
    // four resident CTAs of each field per SM, fewer where the field is small
    const size_t want = (count / 8 + 255) / 256, most = (size_t)(4 * (num_sms > 0 ? num_sms : 152));
    const unsigned nb = (unsigned)(want < 1 ? 1 : (want < most ? want : most));
    off_absmax_k<<<dim3(nb, 2), 256, 0, st>>>((const unsigned short *)f, (const unsigned short *)g,
                                              count, maxbits);
    const OffBuf cur = off_view(f, g, N);
    if (codec == OFFSET_F16)
        off_target_k<CodecF16><<<1, 1, 0, st>>>(cur, maxbits, target);
    else
        off_target_k<CodecBF16><<<1, 1, 0, st>>>(cur, maxbits, target);
    return cudaGetLastError();
}

}  // namespace wblbm
