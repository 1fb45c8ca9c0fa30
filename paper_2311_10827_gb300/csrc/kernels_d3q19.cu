// D3Q19 kernels of the well-balanced phase-field LBM.  The paper works in 2D
// (D2Q9); the 3D form keeps its equilibria (Eqs. H_i, G_i, Siu), sources
// (Eqs. F_i, GGi), moments and isotropic stencils (Eqs. gradient, Laplace)
// on the standard 19-velocity lattice (weights 1/3, 1/18, 1/36; cs^2 = 1/3).
//
// Storage as in 2D: pull scheme, SoA [i][z][y][x], post-collision values at
// their source node.  A step is two passes:
//   1. d3q19_phi_kernel: phi = sum_i f_i pulled (one FP field);
//   2. d3q19_pass32_kernel (FP32, two nodes per thread) or d3q19_pass_kernel
//      (FP64, one): a CTA owns a TX x TY column tile and marches down z; phi
//      planes (tile + 2 halo, read from the phi field, mostly L2) and mu planes
//      (tile + 1) live in shared-memory rings; each node pulls its 19 + 19
//      populations, recovers the moments and collides.
// HBM traffic per node of the FP32 form: 84 B for pass 1, 324 B for pass 2.  As
// in 2D, FP32 storage keeps the rest population as a compensated pair hi + lo
// (lo in population slot 19) so that its small per-step changes are not lost.
#include <float.h>
#include <math.h>

#include "d3q19_lattice.cuh"
#include "launch.cuh"
#include "lbm_internal.h"
#include "rcp64.cuh"
#include "pair32.cuh"

namespace wblbm {
namespace {

using namespace d3;

// phi = sum_i f_i(x - c_i): rest population last, moving ones in fixed pairs
// grid (ceil(nx / PHI_TX), ny, nz): one thread per node of a row
constexpr int PHI_TX = 128;
template <typename T>
__global__ void __launch_bounds__(PHI_TX)
    d3q19_phi_kernel(const StepParams<T> P, const T *__restrict__ f, T *__restrict__ phi)
{
    const int bx = pdl_wait(blockIdx.x);
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x = bx * PHI_TX + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= nx) return;
    const unsigned N = (unsigned)P.N;
    const Nb b = make_nb(x, y, z, nx, ny, nz);
    const unsigned n = b.at(0, 0, 0);
    T v[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) v[i] = __ldg(f + (i * N + b.at(-c3x(i), -c3y(i), -c3z(i))));
    T s = sizeof(T) == 4 ? __ldg(f + (19u * N + n)) : T(0);  // low word of the rest pair
#pragma unroll
    for (int i = 1; i < 19; i += 2) s += v[i] + v[i + 1];
    phi[n] = v[0] + s;
}

// One CTA's diagnostics partial from its NT threads' values (all of them call it)
template <int NT>
__device__ __forceinline__ void write_partial3(int tid, double d_phi, double d_E, double d_u2,
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

// The FP64 pass: one node per thread.  The FP64 pipe bounds it (one warp
// operation per 16 cycles and SM), so the update is written for the fewest
// operations: sums and differences of opposite populations serve the moments,
// diagonal differences serve two gradient components, a reciprocal is three
// operations, and a collision is one or two multiply-adds per population on
// coefficients formed once per node (INCG: g relaxes by increments, INCR_G).
// 100 x 75 x 130 1447 -> 1060 us per step (1108 with tau_g > 2), 160^3 4.06 -> 2.96 ms
// (3.10).
template <int PASS, bool INCG>
__global__ void __launch_bounds__(TX3 *TY3)
    d3q19_pass_kernel(const StepParams<double> P, PassArgs a, const double *__restrict__ phif,
                      int planes)
{
    using T = double;
    constexpr int PX = TX3 + 4, PY = TY3 + 4, PA = PX * PY;  // phi plane (halo 2)
    constexpr int MX = TX3 + 2, MY = TY3 + 2, MA = MX * MY;  // mu plane (halo 1)
    constexpr int RP = 5, RM = 3;
    __shared__ T phs[RP * PA];
    __shared__ T mus[RM * MA];

    const int bx = pdl_wait(blockIdx.x);
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const unsigned N = (unsigned)P.N;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX3 + tx;
    const int x0 = bx * TX3, y0 = blockIdx.y * TY3;
    const int z0 = blockIdx.z * planes, zend = min(z0 + planes, nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool col_ok = x < nx && y < ny;
    const T *__restrict__ fsrc = static_cast<const T *>(a.f_src);
    const T *__restrict__ gsrc = static_cast<const T *>(a.g_src);
    const unsigned plane = (unsigned)nx * ny;

    auto pslot = [&](int zz) { return (zz - z0 + 2) % RP; };  // zz >= z0 - 2
    auto mslot = [&](int zz) { return (zz - z0 + 1) % RM; };  // zz >= z0 - 1

    // grids narrower than a tile plus halo wrap by division (uniform flags)
    const bool smx = nx < PX + 2, smy = ny < PY + 2, smz = nz < 8;
    auto load_phi_plane = [&](int zz) {
        T *dst = phs + pslot(zz) * PA;
        const unsigned zo = (unsigned)wrapc(zz, nz, smz) * plane;
        for (int q = tid; q < PA; q += TX3 * TY3) {
            const int lx = q % PX, ly = q / PX;
            const unsigned xx = wrapc(x0 - 2 + lx, nx, smx), yy = wrapc(y0 - 2 + ly, ny, smy);
            dst[q] = phif[zo + yy * nx + xx];
        }
    };
    // Eq. chemical_potencial with Eq. Laplace on D3Q19:
    // lap = (1/3) sum_faces (phi_n - phi) + (1/6) sum_edges (phi_n - phi)
    auto mu_plane = [&](int zz) {
        const T *pm = phs + pslot(zz - 1) * PA, *p0 = phs + pslot(zz) * PA,
                *pp = phs + pslot(zz + 1) * PA;
        T *dst = mus + mslot(zz) * MA;
        for (int q = tid; q < MA; q += TX3 * TY3) {
            const int lx = q % MX + 1, ly = q / MX + 1;  // phi plane coordinates
            const int c = ly * PX + lx;
            const T v = p0[c];
            const T fa = (p0[c + 1] - v) + (p0[c - 1] - v) + (p0[c + PX] - v) + (p0[c - PX] - v) +
                         (pp[c] - v) + (pm[c] - v);
            const T ed = ((p0[c + PX + 1] - v) + (p0[c + PX - 1] - v) + (p0[c - PX + 1] - v) +
                          (p0[c - PX - 1] - v)) +
                         ((pp[c + 1] - v) + (pp[c - 1] - v) + (pm[c + 1] - v) + (pm[c - 1] - v)) +
                         ((pp[c + PX] - v) + (pp[c - PX] - v) + (pm[c + PX] - v) + (pm[c - PX] - v));
            const T lap = T(1.0 / 3.0) * fa + T(1.0 / 6.0) * ed;
            dst[q] = T(4) * P.beta * (v - P.phil) * (v - P.phiv) * (v - P.phibar) - P.kappa * lap;
        }
    };
    // 6 times the gradient of Eq. gradient on D3Q19: face differences plus half the
    // edge differences; a and b are the differences along the diagonals of a
    // plane of axes, a + b and a - b its two edge terms
    auto grad6 = [&](const T *m, const T *c0, const T *p, int c, int SX, T out[3]) {
        const T a0 = c0[c + SX + 1] - c0[c - SX - 1], b0 = c0[c - SX + 1] - c0[c + SX - 1];  // x, y
        const T a1 = p[c + 1] - m[c - 1], b1 = m[c + 1] - p[c - 1];                          // x, z
        const T a2 = p[c + SX] - m[c - SX], b2 = m[c + SX] - p[c - SX];                      // y, z
        out[0] = fma(T(0.5), (a0 + b0) + (a1 + b1), c0[c + 1] - c0[c - 1]);
        out[1] = fma(T(0.5), (a0 - b0) + (a2 + b2), c0[c + SX] - c0[c - SX]);
        out[2] = fma(T(0.5), (a1 - b1) + (a2 - b2), p[c] - m[c]);
    };

    double d_phi = 0.0, d_E = 0.0, d_u2 = 0.0, d_mumin = DBL_MAX, d_mumax = -DBL_MAX,
           d_bud = 0.0, d_bad = 0.0;

    for (int q = 0; q < 5; ++q) load_phi_plane(z0 - 2 + q);
    __syncthreads();
    mu_plane(z0 - 1);
    mu_plane(z0);
    mu_plane(z0 + 1);
    __syncthreads();

    // Plane zz + 3 of phi travels through registers while plane zz is
    // updated, so its loads overlap the node's own pulls (one exposed memory
    // latency per plane).  Ring use during the update of plane zz: phi planes
    // zz-1..zz+1 (read), zz+3 (written: a fifth slot); mu planes zz-1..zz+1.
    constexpr int PPT = (PA + TX3 * TY3 - 1) / (TX3 * TY3);
    const unsigned xw = col_ok ? (unsigned)x : 0, yw = col_ok ? (unsigned)y : 0;
    Nb b = make_nb(xw, yw, z0, nx, ny, nz);
    for (int zz = z0; zz < zend; ++zz) {
        T pre[PPT];
        {
            const unsigned zo = (unsigned)wrapc(zz + 3, nz, smz) * plane;
#pragma unroll
            for (int k = 0; k < PPT; ++k) {
                const int q = tid + k * TX3 * TY3;
                if (q < PA) {
                    const unsigned xx = wrapc(x0 - 2 + q % PX, nx, smx),
                                   yy = wrapc(y0 - 2 + q / PX, ny, smy);
                    pre[k] = phif[zo + yy * nx + xx];
                }
            }
        }
        if (col_ok) {
        nb_plane(b, zz, nx, ny, nz);
        const unsigned n = b.at(0, 0, 0);
        T fv[19], gv[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const unsigned src = b.at(-c3x(i), -c3y(i), -c3z(i));
            fv[i] = __ldg(fsrc + (i * N + src));
            gv[i] = __ldg(gsrc + (i * N + src));
        }
        T Sprev = T(0);
        if (PASS & (PASS_STATE | PASS_DIAG)) Sprev = __ldcs(static_cast<const T *>(a.S) + n);

        // opposite of direction i
        auto opp = [](int i) {
            return (i <= 6) ? (i % 2 ? i + 1 : i - 1)
                            : (i <= 10 ? 17 - i : (i <= 14 ? 25 - i : 33 - i));
        };
        T snz = fv[1] + fv[2], sg = gv[1] + gv[2];
        T j3[3] = {gv[1] - gv[2], gv[3] - gv[4], gv[5] - gv[6]};
#pragma unroll
        for (int i = 3; i < 19; ++i) {
            const int o = opp(i);
            if (o < i) continue;  // each pair once, from its first member
            snz += fv[i] + fv[o];
            sg += gv[i] + gv[o];
            if (i <= 6) continue;
            const T d = gv[i] - gv[o];
            if (c3x(i)) j3[0] = c3x(i) > 0 ? j3[0] + d : j3[0] - d;
            if (c3y(i)) j3[1] = c3y(i) > 0 ? j3[1] + d : j3[1] - d;
            if (c3z(i)) j3[2] = c3z(i) > 0 ? j3[2] + d : j3[2] - d;
        }
        const T phi = fv[0] + snz;
        const int cp = (ty + 2) * PX + (tx + 2), cm = (ty + 1) * MX + (tx + 1);
        const T *mz = mus + mslot(zz) * MA;
        const T mu = mz[cm];
        T q[3], gm[3];  // 6 grad(phi), 6 grad(mu)
        grad6(phs + pslot(zz - 1) * PA, phs + pslot(zz) * PA, phs + pslot(zz + 1) * PA, cp, PX, q);
        grad6(mus + mslot(zz - 1) * MA, mz, mus + mslot(zz + 1) * MA, cm, MX, gm);

        T F[3], u[3];
        const T dphi = phi - P.phiv;
        const T rho = fma(P.drho, dphi, P.rhov);
        const T taug = fma(T(3) * P.dnu, dphi, fma(T(3), P.nuv, T(0.5)));
        const T irho = rcp64(rho), itg = rcp64(taug);
        const T f6 = T(-1.0 / 6.0) * phi;
        T uu = T(0), S6 = T(0);  // S6: 6 u.grad(phi)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            F[d] = fma(f6, gm[d], P.G[d]);
            u[d] = fma(T(0.5), F[d], j3[d]) * irho;
            uu = d == 0 ? u[d] * u[d] : fma(u[d], u[d], uu);
            S6 = d == 0 ? u[d] * q[d] : fma(u[d], q[d], S6);
        }
        const T S = T(1.0 / 6.0) * S6, ruu = rho * uu;
        // p = cs2/(1 - w0) [sum_{i!=0} g_i + u.grad(rho)/2 + rho s_0], cs2/(1-w0) = 1/2,
        // rho s_0 = -(1/2) rho |u|^2
        const T p = T(0.5) * fma(T(-0.5), ruu, fma(T(0.5) * P.drho, S, sg));

        if (PASS & PASS_DIAG) {
            const double u2 = (double)uu;
            d_phi += (double)phi;
            d_E += 0.5 * (double)rho * u2;
            d_u2 = fmax(d_u2, u2);
            d_mumin = fmin(d_mumin, (double)mu);
            d_mumax = fmax(d_mumax, (double)mu);
            d_bud += 1.5 * (double)S - 0.5 * (double)Sprev;
            if (!isfinite((double)phi) || !isfinite((double)p) || !isfinite(u2) ||
                !isfinite((double)mu))
                d_bad = 1.0;
        }
        if (PASS & PASS_MACROS) {
            if (a.out_phi) a.out_phi[n] = (double)phi;
            if (a.out_p) a.out_p[n] = (double)p;
            if (a.out_mu) a.out_mu[n] = (double)mu;
            if (a.out_u) {
                a.out_u[n] = (double)u[0];
                a.out_u[(size_t)N + n] = (double)u[1];
                a.out_u[2 * (size_t)N + n] = (double)u[2];
            }
        }
        if (PASS & PASS_STATE) {
            T *__restrict__ fd = static_cast<T *>(a.f_dst);
            T *__restrict__ gd = static_cast<T *>(a.g_dst);
            __stcs(static_cast<T *>(a.S) + n, S);
            // CH population: b = -5/2, -1, 1/2 (rest, face, edge) for D = 3;
            // f* = f (1 - 1/tau_f) + w_i z + w_i b_i Sh, z = alpha mu / tau_f
            const T Sh = fma(T(1.5), S, T(-0.5) * Sprev);
            const T itf = P.inv_tauf, omf = T(1) - itf, z = (itf * P.alpha) * mu;
            // (the rest population's increment first: one rounding at its size)
            __stcs(fd + n, fv[0] + fma(itf, snz, fma(T(-2.0 / 3.0), z, T(-5.0 / 6.0) * Sh)));
            const T ka = T(1.0 / 18.0) * (z - Sh), ke = T(1.0 / 36.0) * fma(T(0.5), Sh, z);
            auto collide_f = [&](auto inc) {
#pragma unroll
                for (int i = 1; i < 19; ++i)
                    __stcs(fd + (i * N + n), relax64<inc.value>(fv[i], itf, omf, i <= 6 ? ka : ke));
            };
            if (P.incr & INCR_F)
                collide_f(std::true_type{});
            else
                collide_f(std::false_type{});
            // hydrodynamic population, pairs of opposite directions: even part
            // E = w [A/tau_g + c.u (4.5 rho/tau_g c.u + 3 k c.grad rho)], odd part
            // O = w [3 rho/tau_g c.u + 3 k c.F], k = 1 - 1/(2 tau_g); coefficients at the
            // faces' weight, the edges take half at the end
            const T p3 = T(3) * p, A = fma(T(-1.5), ruu, p3), omg = T(1) - itg;
            const T itw = T(1.0 / 18.0) * itg, kw = fma(T(-0.5), itw, T(1.0 / 18.0));
            const T e0 = itw * A, ri = rho * itw, e1 = T(4.5) * ri, o1 = T(3) * ri;
            const T e2 = (T(0.5) * P.drho) * kw, o2 = T(3) * kw;
            auto dot = [](int cx, int cy, int cz, const T v[3]) -> T {
                T s = cx ? (cx > 0 ? v[0] : -v[0]) : (cy ? (cy > 0 ? v[1] : -v[1]) : (cz > 0 ? v[2] : -v[2]));
                if (cx && cy) s = cy > 0 ? s + v[1] : s - v[1];
                if ((cx || cy) && cz) s = cz > 0 ? s + v[2] : s - v[2];
                return s;
            };
            __stcs(gd + n, relax64<INCG>(gv[0], itg, omg, itg * fma(T(1.0 / 3.0), A, -p3)));
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                const int o = opp(i);
                if (o < i) continue;
                const T cu = dot(c3x(i), c3y(i), c3z(i), u), cF = dot(c3x(i), c3y(i), c3z(i), F);
                const T cq = dot(c3x(i), c3y(i), c3z(i), q);
                const T E = fma(cu, fma(e2, cq, e1 * cu), e0), O = fma(o2, cF, o1 * cu);
                const T w = i <= 6 ? T(1) : T(0.5);
                __stcs(gd + (i * N + n), relax64<INCG>(gv[i], itg, omg, w * (E + O)));
                __stcs(gd + (o * N + n), relax64<INCG>(gv[o], itg, omg, w * (E - O)));
            }
        }
        }  // col_ok
        {
            T *d = phs + pslot(zz + 3) * PA;
#pragma unroll
            for (int k = 0; k < PPT; ++k) {
                const int q = tid + k * TX3 * TY3;
                if (q < PA) d[q] = pre[k];
            }
        }
        __syncthreads();
        mu_plane(zz + 2);
        __syncthreads();
    }

    if (PASS & PASS_DIAG)
        write_partial3<TX3 * TY3>(tid, d_phi, d_E, d_u2, d_mumin, d_mumax, d_bud, d_bad,
                                  a.partials + (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + bx);
}

// The FP32 pass: two nodes adjacent in x per thread (TXP x TY3 threads), their
// arithmetic on the paired FP32 datapath, 64-bit loads and stores of both
// where rows are even (EVEN) and the pull has no x component.
// What bounds it: HBM on large grids (408 B per node with the phi pass, at 90%
// of the copy bandwidth), the latency of a plane on small ones.  719
// instructions per node against 1192 with one node per thread, three CTAs of
// 128 threads per SM (four, at 128 registers: 2% slower at 512^3).  Measured:
// 64^3 24.0 -> 20.2 us per step, 512^3 runs 10.6 -> 9.7 ms per step.  Not kept:
// phi summed inside this kernel for the plane three ahead (no phi pass): the
// populations it read came back from HBM again for half of the update's pulls
// (205 against 168 B read per node), 512^3 9.58 against 8.92 ms per step, 64^3
// 27.1 against 19.6 us.
template <int PASS, bool EVEN>
__global__ void __launch_bounds__(PAIR_NT, 3)
    d3q19_pass32_kernel(const StepParams<float> P, PassArgs a, const float *__restrict__ phif,
                        int planes)
{
    constexpr int PX = TX3 + 4, PY = TY3 + 4, PA = PX * PY;  // phi plane (halo 2)
    constexpr int MX = TX3 + 4, MY = TY3 + 2, MA = MX * MY;  // mu plane (halo 1; 2 stored in x)
    constexpr int MW = TX3 + 2, MN = MW * MY;                // nodes of a mu plane
    constexpr int RP = 5, RM = 3;
    __shared__ __align__(16) float phs[RP * PA];
    __shared__ __align__(16) float mus[RM * MA];

    const int bx = pdl_wait(blockIdx.x);
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const unsigned N = (unsigned)P.N;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TXP + tx;
    const int x0 = bx * TX3, y0 = blockIdx.y * TY3;
    const int z0 = blockIdx.z * planes, zend = min(z0 + planes, nz);
    const int x = x0 + 2 * tx, y = y0 + ty;
    const bool okA = x < nx && y < ny, okB = EVEN ? okA : (x + 1 < nx && y < ny);
    const unsigned plane = (unsigned)nx * ny;
    const float *__restrict__ fsrc = static_cast<const float *>(a.f_src);
    const float *__restrict__ gsrc = static_cast<const float *>(a.g_src);

    // grids narrower than a tile plus halo wrap by division (uniform flags)
    const bool smx = nx < PX + 2, smy = ny < PY + 2, smz = nz < 8;
    // this thread's elements of a phi plane and nodes of a mu plane
    constexpr int KP = (PA + PAIR_NT - 1) / PAIR_NT, KM = (MN + PAIR_NT - 1) / PAIR_NT;
    unsigned poff[KP];
    int mring[KM];
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        const int q = tid + k * PAIR_NT;
        poff[k] = (unsigned)wrapc(y0 - 2 + q / PX, ny, smy) * nx + wrapc(x0 - 2 + q % PX, nx, smx);
    }
#pragma unroll
    for (int k = 0; k < KM; ++k) {
        const int q = tid + k * PAIR_NT;
        mring[k] = q / MW * MX + q % MW + 1;
    }
    auto wrapr = [](int v, int n) { return v >= n ? v - n : v; };
    // Eq. chemical_potencial with Eq. Laplace on D3Q19, from the phi slots of the
    // planes below, at and above into mu slot sm:
    // lap = (1/3) sum_faces (phi_n - phi) + (1/6) sum_edges (phi_n - phi)
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

    double d_phi = 0.0, d_E = 0.0, d_u2 = 0.0, d_mumin = DBL_MAX, d_mumax = -DBL_MAX,
           d_bud = 0.0, d_bad = 0.0;

    // equilibrium shift of the source buffer and of the writes (only a time step reads it)
    float a_src = 0.0f, a_dst = 0.0f;
    if (PASS & PASS_STATE) {
        a_src = *a.eqs_src;
        a_dst = *a.eqs_target;
        if (bx == 0 && blockIdx.y == 0 && blockIdx.z == 0 && tid == 0) *a.eqs_dst = a_dst;
    }

    for (int d = 0; d < 5; ++d) {
        const unsigned zo = (unsigned)wrapc(z0 - 2 + d, nz, smz) * plane;
#pragma unroll
        for (int k = 0; k < KP; ++k)
            if (tid + k * PAIR_NT < PA) cp_async4(phs + d * PA + tid + k * PAIR_NT, phif + zo + poff[k]);
    }
    cp_commit();
    cp_wait_all();
    __syncthreads();
    for (int d = 0; d < 3; ++d) mu_plane(d, d + 1, d + 2, d);
    __syncthreads();

    // Plane zz + 3 of phi is copied asynchronously while plane zz is updated.
    // Ring use during the update of plane zz: phi planes zz-1..zz+1 (read),
    // zz+3 (written: a fifth slot); mu planes zz-1..zz+1.
    const unsigned xw = okA ? (unsigned)x : 0, yw = okA ? (unsigned)y : 0;
    Nb b = make_nb((int)xw, (int)yw, z0, nx, ny, nz);
    const unsigned xB = okB ? xw + 1 : 0;  // the second node's column and its +x neighbour
    const unsigned xpp = nx == 1 ? 0u : (unsigned)wrap1((int)xw + 2, nx);
    int sp = 1, sq = 0;  // phi slot of plane zz - 1, mu slot of plane zz - 1
    for (int zz = z0; zz < zend; ++zz) {
        const int sp0 = wrapr(sp + 1, RP), spp = wrapr(sp + 2, RP);
        const int sq0 = wrapr(sq + 1, RM), sqp = wrapr(sq + 2, RM);
        {
            const unsigned zo = (unsigned)wrapc(zz + 3, nz, smz) * plane;
            float *d = phs + wrapr(sp + 4, RP) * PA + tid;
#pragma unroll
            for (int k = 0; k < KP; ++k)
                if (tid + k * PAIR_NT < PA) cp_async4(d + k * PAIR_NT, phif + (zo + poff[k]));
            cp_commit();
        }
        if (okA) {
        nb_plane(b, zz, nx, ny, nz);
        const unsigned row = b.zs[1] + b.ys[1], n = row + xw;
        auto pull = [&](const float *v, int i) -> float2 {
            const unsigned r = i * N + b.zs[1 - c3z(i)] + b.ys[1 - c3y(i)];
            if (c3x(i) == 0 && EVEN) return __ldg(reinterpret_cast<const float2 *>(v + (r + xw)));
            const unsigned ca = c3x(i) > 0 ? b.xs[0] : (c3x(i) < 0 ? b.xs[2] : xw);
            const unsigned cb = c3x(i) > 0 ? xw : (c3x(i) < 0 ? xpp : xB);
            return make_float2(__ldg(v + (r + ca)), __ldg(v + (r + cb)));
        };
        float2 fv[19], gv[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            fv[i] = pull(fsrc, i);
            gv[i] = pull(gsrc, i);
        }
        float2 Sprev = f2(0.0f), lo0;
        if (EVEN)
            lo0 = __ldg(reinterpret_cast<const float2 *>(fsrc + (19u * N + n)));
        else
            lo0 = make_float2(__ldg(fsrc + (19u * N + n)), __ldg(fsrc + (19u * N + row + xB)));
        if (PASS & (PASS_STATE | PASS_DIAG)) {
            const float *S = static_cast<const float *>(a.S);
            if (EVEN)
                Sprev = __ldcs(reinterpret_cast<const float2 *>(S + n));
            else
                Sprev = make_float2(__ldcs(S + n), __ldcs(S + (row + xB)));
        }

        float2 snz = add2(fv[1], fv[2]), sg = add2(gv[1], gv[2]);
#pragma unroll
        for (int i = 3; i < 19; i += 2) {
            snz = add2(snz, add2(fv[i], fv[i + 1]));
            sg = add2(sg, add2(gv[i], gv[i + 1]));
        }
        const float2 phi = add2(fv[0], add2(lo0, snz));
        const int cp = (ty + 2) * PX + 2 * tx + 2, c0 = (ty + 1) * MX + 2 * tx + 2;
        const float *m0 = mus + sq0 * MA;
        const float2 mu = pair_at(m0, c0, true);
        float2 gp[3], gm[3];
        grad3_pair(phs + sp * PA, phs + sp0 * PA, phs + spp * PA, cp, PX, gp);
        grad3_pair(mus + sq * MA, m0, mus + sqp * MA, c0, MX, gm);

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
        // p = cs2/(1 - w0) [sum_{i!=0} g_i + u.grad(rho)/2 + rho s_0], cs2/(1-w0) = 1/2,
        // rho s_0 = -(1/2) rho |u|^2
        const float2 p =
            mul2(f2(0.5f), fma2(mul2(f2(-0.5f), rho), uu, fma2(f2(0.5f), ugr, sg)));

        if (PASS & PASS_DIAG) {
            auto acc = [&](float ph, float rh, float u2f, float m, float Sn, float So, float pp) {
                const double u2 = (double)u2f;
                d_phi += (double)ph;
                d_E += 0.5 * (double)rh * u2;
                d_u2 = fmax(d_u2, u2);
                d_mumin = fmin(d_mumin, (double)m);
                d_mumax = fmax(d_mumax, (double)m);
                d_bud += 1.5 * (double)Sn - 0.5 * (double)So;
                if (!isfinite(ph) || !isfinite(pp) || !isfinite(u2f) || !isfinite(m)) d_bad = 1.0;
            };
            acc(phi.x, rho.x, uu.x, mu.x, S.x, Sprev.x, p.x);
            if (okB) acc(phi.y, rho.y, uu.y, mu.y, S.y, Sprev.y, p.y);
        }
        if (PASS & PASS_MACROS) {
            auto put = [&](double *o, float2 v) {
                o[n] = (double)v.x;
                if (okB) o[n + 1] = (double)v.y;
            };
            if (a.out_phi) put(a.out_phi, phi);
            if (a.out_p) put(a.out_p, p);
            if (a.out_mu) put(a.out_mu, mu);
            if (a.out_u) {
#pragma unroll
                for (int d = 0; d < 3; ++d) put(a.out_u + d * (size_t)N, u[d]);
            }
        }
        if (PASS & PASS_STATE) {
            float *__restrict__ fd = static_cast<float *>(a.f_dst);
            float *__restrict__ gd = static_cast<float *>(a.g_dst);
            auto put = [&](float *o, float2 v) {
                if (EVEN) {
                    __stcs(reinterpret_cast<float2 *>(o + n), v);
                } else {
                    __stcs(o + n, v.x);
                    if (okB) __stcs(o + n + 1, v.y);
                }
            };
            put(static_cast<float *>(a.S), S);
            // CH population: b = -5/2, -1, 1/2 (rest, face, edge) for D = 3
            const float2 Sh = fma2(f2(1.5f), S, mul2(f2(-0.5f), Sprev));
            const float2 am = fma2(f2(P.alpha), mu, f2(-a_src));  // in the source's shifted variables
            const float dsh = a_src - a_dst;                      // move the writes to the target shift
            const float2 itf = f2(P.inv_tauf);
            {
                const float2 q = fma2(f2(-(2.0f / 3.0f)), am, snz);
                const float2 d0 = fma2(f2(-(5.0f / 6.0f)), Sh,
                                       fma2(q, itf, f2(-(2.0f / 3.0f) * dsh)));
                const float2 sl = add2(lo0, d0);  // exact two-sum on the high word
                const float2 hi = add2(fv[0], sl);
                const float2 bp = sub2(hi, fv[0]);
                put(fd, hi);
                put(fd + 19u * N, add2(sub2(fv[0], sub2(hi, bp)), sub2(sl, bp)));
            }
            // each population moves by its own small increment (as in 2D: the
            // increments sum to sum_i F_i up to unbiased rounding)
            const float2 ea = mul2(f2(1.0f / 18.0f), am), ee = mul2(f2(1.0f / 36.0f), am);
            const float2 sa = fma2(f2(-1.0f / 18.0f), Sh, f2((1.0f / 18.0f) * dsh));
            const float2 se = fma2(f2(1.0f / 72.0f), Sh, f2((1.0f / 36.0f) * dsh));
#pragma unroll
            for (int i = 1; i < 19; ++i)
                put(fd + i * N,
                    add2(fv[i], fma2(sub2(i <= 6 ? ea : ee, fv[i]), itf, i <= 6 ? sa : se)));
            // hydrodynamic population, pairs of opposite directions (as in 2D)
            const float2 kg = fma2(f2(-0.5f), itg, f2(1.0f));
            const float2 p3 = mul2(f2(3.0f), p);
            const float2 A = fma2(mul2(f2(-1.5f), rho), uu, p3);
            put(gd, fma2(sub2(sub2(mul2(f2(1.0f / 3.0f), A), p3), gv[0]), itg, gv[0]));
            const float2 r45 = mul2(f2(4.5f), rho);
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                const int o = (i <= 6) ? (i % 2 ? i + 1 : i - 1)
                                       : (i <= 10 ? 17 - i : (i <= 14 ? 25 - i : 33 - i));
                if (o < i) continue;  // each pair once, from its first member
                const float w = (float)w3(i);
                const float2 cu = dot_c(c3x(i), c3y(i), c3z(i), u[0], u[1], u[2]);
                const float2 cF = dot_c(c3x(i), c3y(i), c3z(i), F[0], F[1], F[2]);
                const float2 cg = dot_c(c3x(i), c3y(i), c3z(i), gr[0], gr[1], gr[2]);
                const float2 es = mul2(f2(w), fma2(mul2(r45, cu), cu, A));
                const float2 ea_ = mul2(mul2(f2(3.0f * w), rho), cu);
                const float2 wk = mul2(f2(3.0f * w), kg);
                const float2 Gs = mul2(mul2(wk, cu), cg), Ga = mul2(wk, cF);
                put(gd + i * N, add2(gv[i], fma2(sub2(add2(es, ea_), gv[i]), itg, add2(Gs, Ga))));
                put(gd + o * N, add2(gv[o], fma2(sub2(sub2(es, ea_), gv[o]), itg, sub2(Gs, Ga))));
            }
        }
        }  // okA
        cp_wait_all();
        __syncthreads();
        // phi planes zz + 1 .. zz + 3 -> mu plane zz + 2 in the slot of zz - 1
        mu_plane(spp, wrapr(sp + 3, RP), wrapr(sp + 4, RP), sq);
        __syncthreads();
        sp = sp0;
        sq = sq0;
    }

    if (PASS & PASS_DIAG)
        write_partial3<PAIR_NT>(tid, d_phi, d_E, d_u2, d_mumin, d_mumax, d_bud, d_bad,
                                a.partials + (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + bx);
}

// ------------------------------------------------------------ initial state

// f_i(x, 0) = f_i^eq(phi0(x), mu0(x)) with mu0 in FP64, the value of node x
// stored at x - c_i; g = 0, S = 0.  As in 2D each node forms its two distinct
// values w_i alpha mu once and stores them 18 times, because the FP64 pipe
// bounds the kernel (64^3 FP32: 60 -> 34 us against a second pass that formed
// them where they are stored).
template <typename T>
__global__ void __launch_bounds__(256)
    d3q19_init_k(const StepParams<double> P, const double *__restrict__ phi, T *__restrict__ f,
                 T *__restrict__ g, T *__restrict__ S)
{
    const unsigned N = (unsigned)P.N, n = blockIdx.x * 256u + threadIdx.x;
    if (n >= N) return;
    const unsigned nx = P.nx, ny = P.ny;
    const unsigned r = n / nx;
    const Nb b = make_nb((int)(n - r * nx), (int)(r % ny), (int)(r / ny), P.nx, P.ny, P.nz);
    const double c = __ldg(phi + n);
    const double am = P.alpha * mu_of_field(P, phi, b, c);
    const double f0 = c - (1.0 - w3(0)) * am;
    f[n] = (T)f0;
    if (sizeof(T) == 4) f[19u * N + n] = (T)(f0 - (double)(T)f0);
    const T va = (T)(w3(1) * am), ve = (T)(w3(7) * am);
#pragma unroll
    for (int i = 1; i < 19; ++i)
        f[i * N + b.at(-c3x(i), -c3y(i), -c3z(i))] = i <= 6 ? va : ve;
#pragma unroll
    for (int i = 0; i < 19; ++i) g[i * N + n] = T(0);
    S[n] = T(0);
}

template <typename T>
__global__ void d3q19_get_state_k(StepParams<double> P, const T *__restrict__ f,
                                  const T *__restrict__ g, const T *__restrict__ S,
                                  const float *eqs, double *fo, double *go, double *So)
{
    const size_t N = (size_t)P.N;
    const size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x = (int)(n % nx), y = (int)((n / nx) % ny), z = (int)(n / ((size_t)nx * ny));
    const Nb b = make_nb(x, y, z, nx, ny, nz);
    for (int i = 0; i < 19; ++i) {
        const unsigned m = b.at(-c3x(i), -c3y(i), -c3z(i));
        double fv = (double)f[i * N + m];
        if (sizeof(T) == 4 && i == 0) fv += (double)f[19 * N + m];
        if (sizeof(T) == 4) fv += (i == 0 ? -(2.0 / 3.0) : w3(i)) * (double)*eqs;  // equilibrium shift
        if (fo) fo[i * N + n] = fv;
        if (go) go[i * N + n] = (double)g[i * N + m];
    }
    if (So) So[n] = (double)S[n];
}

template <typename T>
__global__ void d3q19_set_state_k(StepParams<double> P, T *__restrict__ f, T *__restrict__ g,
                                  T *__restrict__ S, const double *fi, const double *gi,
                                  const double *Si)
{
    const size_t N = (size_t)P.N;
    const size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x = (int)(n % nx), y = (int)((n / nx) % ny), z = (int)(n / ((size_t)nx * ny));
    const Nb b = make_nb(x, y, z, nx, ny, nz);
    for (int i = 0; i < 19; ++i) {
        const unsigned m = b.at(c3x(i), c3y(i), c3z(i));
        const double v = fi[i * N + m];
        f[i * N + n] = (T)v;
        if (sizeof(T) == 4 && i == 0) f[19 * N + n] = (T)(v - (double)(T)v);
        g[i * N + n] = (T)gi[i * N + m];
    }
    S[n] = (T)Si[n];
}

template <typename T, int PASS>
cudaError_t launch3(const void *params, const PassArgs &a, const LaunchShape &s, void *phi,
                    cudaStream_t st)
{
    const StepParams<T> &P = *static_cast<const StepParams<T> *>(params);
    const dim3 grid(s.grid_x, s.grid_y, s.nblocks / (s.grid_x * s.grid_y));
    const dim3 pg((P.nx + PHI_TX - 1) / PHI_TX, P.ny, P.nz);
    const cudaError_t e = launch_pdl(d3q19_phi_kernel<T>, pg, PHI_TX, 0, st, P,
                                     static_cast<const T *>(a.f_src), static_cast<T *>(phi));
    if (e != cudaSuccess) return e;
    if constexpr (sizeof(T) == 4) {
        const dim3 block(TXP, TY3);
        if (P.nx % 2 == 0)
            return launch_pdl(d3q19_pass32_kernel<PASS, true>, grid, block, 0, st, P, a,
                              static_cast<const float *>(phi), s.rows);
        return launch_pdl(d3q19_pass32_kernel<PASS, false>, grid, block, 0, st, P, a,
                          static_cast<const float *>(phi), s.rows);
    } else {
        if constexpr (PASS & PASS_STATE)
            if (P.incr & INCR_G)
                return launch_pdl(d3q19_pass_kernel<PASS, true>, grid, dim3(TX3, TY3), 0, st, P, a,
                                  static_cast<const T *>(phi), s.rows);
        return launch_pdl(d3q19_pass_kernel<PASS, false>, grid, dim3(TX3, TY3), 0, st, P, a,
                          static_cast<const T *>(phi), s.rows);
    }
}

template <typename T>
cudaError_t pass3_t(int pass, const void *params, const PassArgs &a, const LaunchShape &s,
                    void *phi, cudaStream_t st)
{
    switch (pass) {
    case PASS_STATE: return launch3<T, PASS_STATE>(params, a, s, phi, st);
    case PASS_STATE | PASS_DIAG: return launch3<T, PASS_STATE | PASS_DIAG>(params, a, s, phi, st);
    case PASS_MACROS: return launch3<T, PASS_MACROS>(params, a, s, phi, st);
    case PASS_DIAG: return launch3<T, PASS_DIAG>(params, a, s, phi, st);
    case PASS_MACROS | PASS_DIAG: return launch3<T, PASS_MACROS | PASS_DIAG>(params, a, s, phi, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

LaunchShape d3q19_shape(int nx, int ny, int nz, int num_sms, int ctas_per_sm)
{
    LaunchShape s;
    s.variant = 0;
    s.grid_x = (nx + TX3 - 1) / TX3;
    s.grid_y = (ny + TY3 - 1) / TY3;
    // Split z into gz marches of `planes` planes.  A march takes about planes + 2
    // planes of work (it starts by filling its rings), and CTAs that share an SM
    // hide part of each other's waits: two take 1.3 times one's time, three 1.6
    // (FP32, 64^3: 256 CTAs of 4 planes 16.7 us, 352 of 3 planes 17.2 us; the FP64
    // pass has one CTA per SM, so that k of them take k times one's).  An SM works
    // through its share of the CTAs, `occ` at a time; pick the split with the
    // least time.  Against counting waves of CTAs with marches of at least four
    // planes, over 26 shapes from 24^3 to 320 x 320 x 24 in each of the four formats:
    // none more than 0.3% slower, 24^3 1.4x (FP64 1.7x), 321 x 24 x 25 1.37x.
    const long long cols = (long long)s.grid_x * s.grid_y;
    const long long occ = ctas_per_sm > 0 ? ctas_per_sm : 2, sms = num_sms > 0 ? num_sms : 152;
    auto share = [](long long k) { return k == 0 ? 0.0 : 1.0 + 0.3 * (double)(k - 1); };
    double best = -1.0;
    long long best_gz = 1;
    const int gz_max = nz / 2 > 1 ? nz / 2 : 1;
    for (int gz = 1; gz <= gz_max; ++gz) {
        const long long planes = (nz + gz - 1) / gz;
        const long long k = (cols * ((nz + planes - 1) / planes) + sms - 1) / sms;  // CTAs per SM
        const double cost = (double)(planes + 2) * ((double)(k / occ) * share(occ) + share(k % occ));
        if (best < 0.0 || cost < best) {
            best = cost;
            best_gz = gz;
        }
    }
    const int planes = (nz + (int)best_gz - 1) / (int)best_gz;
    s.rows = planes;
    s.nblocks = (int)(cols * ((nz + planes - 1) / planes));
    return s;
}

int d3q19_ctas_per_sm(int precision)
{
    int n = 0;
    cudaError_t e = precision == 0
                        ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                              &n, d3q19_pass_kernel<PASS_STATE, false>, TX3 * TY3, 0)
                        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                              &n, d3q19_pass32_kernel<PASS_STATE, true>, PAIR_NT, 0);
    return e == cudaSuccess && n > 0 ? n : 2;
}

cudaError_t d3q19_pass(int precision, int pass, const void *params, const PassArgs &a,
                       const LaunchShape &s, void *phi_work, cudaStream_t st)
{
    return precision == 0 ? pass3_t<double>(pass, params, a, s, phi_work, st)
                          : pass3_t<float>(pass, params, a, s, phi_work, st);
}

cudaError_t d3q19_init(int precision, const void *params, const double *phi0, void *f, void *g,
                       void *S, cudaStream_t st)
{
    const StepParams<double> &P = *static_cast<const StepParams<double> *>(params);
    const unsigned nb = (unsigned)((P.N + 255) / 256);
    if (precision == 0)
        d3q19_init_k<double><<<nb, 256, 0, st>>>(P, phi0, (double *)f, (double *)g, (double *)S);
    else
        d3q19_init_k<float><<<nb, 256, 0, st>>>(P, phi0, (float *)f, (float *)g, (float *)S);
    return cudaGetLastError();
}

cudaError_t d3q19_get_state(int precision, const void *params, const void *f, const void *g,
                            const void *S, const float *eqs, double *fo, double *go, double *So,
                            cudaStream_t st)
{
    const StepParams<double> &P = *static_cast<const StepParams<double> *>(params);
    const unsigned nb = (unsigned)((P.N + 255) / 256);
    if (precision == 0)
        d3q19_get_state_k<double><<<nb, 256, 0, st>>>(P, (const double *)f, (const double *)g,
                                                     (const double *)S, eqs, fo, go, So);
    else
        d3q19_get_state_k<float><<<nb, 256, 0, st>>>(P, (const float *)f, (const float *)g,
                                                    (const float *)S, eqs, fo, go, So);
    return cudaGetLastError();
}

cudaError_t d3q19_set_state(int precision, const void *params, void *f, void *g, void *S,
                            const double *fi, const double *gi, const double *Si, cudaStream_t st)
{
    const StepParams<double> &P = *static_cast<const StepParams<double> *>(params);
    const unsigned nb = (unsigned)((P.N + 255) / 256);
    if (precision == 0)
        d3q19_set_state_k<double><<<nb, 256, 0, st>>>(P, (double *)f, (double *)g, (double *)S, fi, gi, Si);
    else
        d3q19_set_state_k<float><<<nb, 256, 0, st>>>(P, (float *)f, (float *)g, (float *)S, fi, gi, Si);
    return cudaGetLastError();
}

}  // namespace wblbm
