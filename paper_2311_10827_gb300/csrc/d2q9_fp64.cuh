// The FP64 tile march of the D2Q9 step.  Internal header of kernels_d2q9.cu.
//
// What bounds it: the FP64 pipe.  GB300 issues one FP64 warp instruction per
// 16 cycles and SM (about 630 G operations/s on the chip), so a node update
// costs its FP64 operations and nothing else: loads, shared memory, index
// arithmetic and barriers hide behind them.  The march is therefore written
// for the fewest FP64 operations, not for bytes or registers:
//  * vertical second differences v = (phi_N - phi) + (phi_S - phi) and first
//    differences d = phi_N - phi_S are formed once per node and shared with
//    the neighbour columns through shared-memory rings: the Laplacian is
//    h + (2/3) v + (1/6)(v_E + v_W) with h the horizontal second difference,
//    and the gradient (1/2)(phi_E - phi_W) + (1/12)(v_E - v_W),
//    (1/3) d + (1/12)(d_E + d_W).  Every term stays a difference of
//    neighbours, so a uniform field still gives exact zeros;
//  * 1/rho and 1/tau_g are three operations each and as accurate as a divide
//    (rcp64; one reciprocal of rho tau_g for both takes as many, and loses an ulp);
//  * each collision is one multiply-add per population (two for relaxation
//    times above 2, see relax64) on coefficients formed once per node and
//    direction class;
//  * the halo columns of both thread rows are one warp's extra work instead
//    of two warps'.
// About 156 FP64 operations per node (165 with tau_g > 2) against about 250 in the
// form shared with the FP32 kernel before.  Measured, us per step: 1024 x 1024
// 498 -> 344 (359 with tau_g > 2; the operations alone take 260 and 275), 512 x 512
// 153 -> 99 (103), 301 x 203 54.9 -> 32.5 (33.7); 128-column tiles were 6% slower.
#pragma once

// shared memory of one FP64 tile march
template <int TX>
struct TileSmem64 {
    static constexpr int RP = 8;        // phi ring: rows t .. t + 3 read, t + 4, t + 5 next
    static constexpr int RV = 4;        // v, d and mu rings: four rows alive
    static constexpr int WP = TX + 4;   // phi, v, d ring width (halo 2)
    static constexpr int WM = TX + 2;   // mu ring width (halo 1)
    static constexpr int NT = TX * 2;
    double phs[RP * WP], vs[RV * WP], ds[RV * WP], mus[RV * WM];
    double red[7][(NT + 31) / 32];
    int bad;
};

// One tile: columns [x0, x0 + TX), rows [y0, yend), marching in direction dir
// (see d2q9_tile, which this replaces for FP64 storage).  INCG: g relaxes by
// increments (INCR_G).
template <int TX, int PASS, bool NC, bool INCG>
__device__ __forceinline__ void d2q9_tile64(TileSmem64<TX> &sm, double *dyn,
                                            const StepParams<double> &P, const PassArgs &a, int x0,
                                            int y0, int yend, int dir, int part, const int tx)
{
    using SM = TileSmem64<TX>;
    constexpr int WP = SM::WP, WM = SM::WM, NT = SM::NT, NW = (NT + 31) / 32;
    constexpr bool NEED_S = (PASS & (PASS_STATE | PASS_DIAG)) != 0;
    double(*const dacc)[NT] = reinterpret_cast<double(*)[NT]>(dyn);
    double(*const facc)[NT] = dacc + 4;
    const int ty = threadIdx.y, lin = ty * TX + tx;
    const int nx = P.nx, ny = P.ny;
    const unsigned N = (unsigned)P.N;
    const bool small = ny < 4;
    const double *__restrict__ fsrc = static_cast<const double *>(a.f_src);
    const double *__restrict__ gsrc = static_cast<const double *>(a.g_src);

    const int xo = x0 + tx;
    const bool col_ok = xo < nx;
    // columns past the grid's last one are needed up to the stencil's reach
    // (two columns); warps wholly beyond it skip the FP64 work
    const bool col_phi = xo < nx + 2;
    const unsigned xO = wrapi(xo, nx), xOm = wrapi(xo - 1, nx), xOp = wrapi(xo + 1, nx);
    // halo work of both thread rows: the last 8 threads, 4 halo columns each
    // (ring index 0, 1, TX + 2, TX + 3); column k of thread row q
    const int hk = lin - (NT - 8);
    const bool halo = hk >= 0;
    const int hq = (hk >> 2) & 1, hc = hk & 3;
    const int jH = hc < 2 ? hc : TX + hc;
    const int cH = x0 - 2 + jH;
    // (a ragged last strip never reads the ring past its own columns + 2)
    const bool halo_phi = halo && cH < nx + 2;
    const unsigned xH = wrapi(cH, nx), xHm = wrapi(cH - 1, nx), xHp = wrapi(cH + 1, nx);
    // mu halo: columns ring index 0 and TX + 1 (phi ring 1 and TX + 2)
    const bool halo_mu = halo && (hc == 1 || hc == 2) && cH < nx + 1;

    const int first = dir > 0 ? y0 : yend - 1;
    const int nout = yend - y0;
    const double beta4 = 4.0 * P.beta;
    const double kap = P.kappa, k23 = P.kappa * (2.0 / 3.0), k16 = P.kappa * (1.0 / 6.0);

    // ring rows of march coordinate m >= -2
    auto prow = [&](int m) { return sm.phs + ((m + 2) & 7) * WP; };
    auto vrow = [&](int m) { return sm.vs + ((m + 4) & 3) * WP; };
    auto drow = [&](int m) { return sm.ds + ((m + 4) & 3) * WP; };
    auto mrow = [&](int m) { return sm.mus + ((m + 4) & 3) * WM; };

    struct Rows {
        unsigned rm, r0, rp;
    };
    auto rows_of = [&](int m) {
        const int row = first + dir * m;
        Rows r;
        r.rm = (unsigned)wrap_row(row - 1, ny, small) * nx;
        r.r0 = (unsigned)wrap_row(row, ny, small) * nx;
        r.rp = (unsigned)wrap_row(row + 1, ny, small) * nx;
        return r;
    };
    // phi rows mb + ty (own columns, keeping the pulls and their sum) and the
    // halo columns of rows mb, mb + 1
    auto phi_rows = [&](int mb, double v[9], double &s) {
        if (col_phi) {
            const Rows r = rows_of(mb + ty);
            pull9<NC>(fsrc, N, r.rm, r.r0, r.rp, xOm, xO, xOp, v);
            s = sum_moving(v);
            prow(mb + ty)[tx + 2] = v[0] + s;
        }
        if (halo_phi) {
            const Rows r = rows_of(mb + hq);
            double h[9];
            pull9<NC>(fsrc, N, r.rm, r.r0, r.rp, xHm, xH, xHp, h);
            prow(mb + hq)[jH] = h[0] + sum_moving(h);
        }
    };
    // v and d (in +y) of one ring element of row m
    auto vd_at = [&](int m, int j) {
        const double *pm = prow(m - dir), *p0 = prow(m), *pp = prow(m + dir);
        const double n = pp[j], s = pm[j], c = p0[j];
        vrow(m)[j] = (n - c) + (s - c);
        drow(m)[j] = n - s;
    };
    auto vd_rows = [&](int mb) {
        if (col_phi) vd_at(mb + ty, tx + 2);
        if (halo_phi) vd_at(mb + hq, jH);
    };
    // Eq. chemical_potencial; j is the phi ring index.  The double-well
    // derivative is left as its three factors: exactly zero in both bulk phases,
    // and relatively accurate beside them (as t (t^2 - (dphi/2)^2), two operations
    // less per node, it carries the rounding of t^2 there)
    auto mu_at = [&](int m, int j) {
        const double *p0 = prow(m), *v = vrow(m);
        const double c = p0[j];
        const double h = (p0[j + 1] - c) + (p0[j - 1] - c);
        double mu = beta4 * (c - P.phil) * (c - P.phiv) * (c - P.phibar);
        mu = fma(-kap, h, mu);
        mu = fma(-k23, v[j], mu);
        mrow(m)[j - 1] = fma(-k16, v[j + 1] + v[j - 1], mu);
    };
    auto mu_rows = [&](int mb) {
        if (xo < nx + 1) mu_at(mb + ty, tx + 2);
        if (halo_mu) mu_at(mb + hq, jH);
    };

    if (PASS & PASS_DIAG) {
#pragma unroll
        for (int q = 0; q < 4; ++q) dacc[q][lin] = 0.0;
        facc[0][lin] = 0.0;
        facc[1][lin] = INFINITY;
        facc[2][lin] = -INFINITY;
        if (lin == 0) sm.bad = 0;  // read after the march's barriers
    }

    // prologue: phi rows -2 .. 1, v, d and mu rows -1, 0
    double fcur[9], fnext[9], scur = 0.0, snext = 0.0;
#pragma unroll
    for (int i = 0; i < 9; ++i) fcur[i] = fnext[i] = 0.0;
    phi_rows(-2, fnext, snext);
    phi_rows(0, fcur, scur);
    __syncthreads();
    vd_rows(-1);
    __syncthreads();
    mu_rows(-1);

    for (int t = 0; t < nout; t += 2) {
        const int m = t + ty;
        const bool out_ok = col_ok && m < nout;
        const Rows r = rows_of(m);
        double gv[9], Sprev = 0.0;
        if (out_ok) {
            pull9<NC>(gsrc, N, r.rm, r.r0, r.rp, xOm, xO, xOp, gv);
            if (NEED_S)
                Sprev = NC ? __ldcs(static_cast<const double *>(a.S) + (r.r0 + xo))
                           : __ldcg(static_cast<const double *>(a.S) + (r.r0 + xo));
        }
        phi_rows(t + 2, fnext, snext);
        __syncthreads();
        vd_rows(t + 1);
        __syncthreads();
        mu_rows(t + 1);
        __syncthreads();
        if (out_ok) {
            const double *p0 = prow(m), *v = vrow(m), *dd = drow(m);
            const double *mm = mrow(m - dir), *m0 = mrow(m), *mp = mrow(m + dir);
            const int j = tx + 2, k = tx + 1;
            const double phi = fcur[0] + scur;
            const double mu = m0[k];
            // q = 2 grad(phi)
            const double qx = fma(1.0 / 6.0, v[j + 1] - v[j - 1], p0[j + 1] - p0[j - 1]);
            const double qy = fma(1.0 / 6.0, dd[j + 1] + dd[j - 1], (2.0 / 3.0) * dd[j]);
            // F = -phi grad(mu) + G with grad(mu) = (1/3)[axis + (1/4) diagonal]
            const double da = mp[k + 1] - mm[k - 1], db = mm[k + 1] - mp[k - 1];
            const double f3 = (-1.0 / 3.0) * phi;
            const double Fx = fma(f3, fma(0.25, da + db, m0[k + 1] - m0[k - 1]), P.G[0]);
            const double Fy = fma(f3, fma(0.25, da - db, mp[k] - mm[k]), P.G[1]);
            const double dphi = phi - P.phiv;
            const double rho = fma(P.drho, dphi, P.rhov);
            const double taug = fma(3.0 * P.dnu, dphi, fma(3.0, P.nuv, 0.5));
            const double irho = rcp64(rho), itg = rcp64(taug);
            // rho u = sum_i c_i g_i + F/2
            const double ga = gv[5] - gv[7], gb = gv[8] - gv[6];
            const double jx = (gv[2] - gv[4]) + (ga + gb), jy = (gv[3] - gv[1]) + (ga - gb);
            const double ux = fma(0.5, Fx, jx) * irho, uy = fma(0.5, Fy, jy) * irho;
            const double S2 = fma(ux, qx, uy * qy);  // 2 u.grad(phi)
            const double uu = fma(ux, ux, uy * uy), ruu = rho * uu;
            // 3p = (9/5)[sum_{i!=0} g_i + u.grad(rho)/2 - (2/3) rho |u|^2]
            const double p3 =
                1.8 * fma(-2.0 / 3.0, ruu, fma(0.25 * P.drho, S2, sum_moving(gv)));

            if (PASS & PASS_DIAG) {
                dacc[0][lin] += phi;
                dacc[1][lin] = fma(0.5, ruu, dacc[1][lin]);
                dacc[2][lin] = fma(0.5, S2, dacc[2][lin]);
                dacc[3][lin] += Sprev;
                facc[0][lin] = fmax(facc[0][lin], uu);
                facc[1][lin] = fmin(facc[1][lin], mu);
                facc[2][lin] = fmax(facc[2][lin], mu);
                if (!isfinite(phi) || !isfinite(p3) || !isfinite(uu) || !isfinite(mu)) sm.bad = 1;
            }
            const unsigned n = r.r0 + xo;
            if (PASS & PASS_MACROS) {
                if (a.out_phi) a.out_phi[n] = phi;
                if (a.out_p) a.out_p[n] = p3 * (1.0 / 3.0);
                if (a.out_mu) a.out_mu[n] = mu;
                if (a.out_u) {
                    a.out_u[n] = ux;
                    a.out_u[(size_t)N + n] = uy;
                }
            }
            if (PASS & PASS_MACROS_T) {
                static_cast<double *>(a.mt_phi)[n] = phi;
                static_cast<double *>(a.mt_p)[n] = p3 * (1.0 / 3.0);
                static_cast<double *>(a.mt_mu)[n] = mu;
                static_cast<double *>(a.mt_u)[n] = ux;
                static_cast<double *>(a.mt_u)[(size_t)N + n] = uy;
            }
            if (PASS & PASS_STATE) {
                double *__restrict__ fd = static_cast<double *>(a.f_dst);
                double *__restrict__ gd = static_cast<double *>(a.g_dst);
                static_cast<double *>(a.S_out)[n] = 0.5 * S2;
                // Eq. BGK with Eqs. H_i, F_i: f* = f (1 - 1/tau_f) + z w_i + w_i b_i Sh,
                // z = alpha mu / tau_f, Sh = 1.5 S - 0.5 S_prev, b = -2, -1/2, 1;
                // the rest population through f_0 - f_0^eq = (5/9) alpha mu - sum f_i,
                // its increment formed first: one rounding at its size, which is phi's
                const double Sh = fma(0.75, S2, -0.5 * Sprev);
                const double itf = P.inv_tauf, omf = 1.0 - itf;
                const double z = (itf * P.alpha) * mu;
                fd[n] = fcur[0] + fma(itf, scur, fma(-5.0 / 9.0, z, (-8.0 / 9.0) * Sh));
                const double ka = (1.0 / 9.0) * fma(-0.5, Sh, z), kd = (1.0 / 36.0) * (z + Sh);
                auto collide_f = [&](auto inc) {
#pragma unroll
                    for (int i = 1; i < 9; ++i)
                        fd[i * N + n] = relax64<inc.value>(fcur[i], itf, omf, i < 5 ? ka : kd);
                };
                if (P.incr & INCR_F)
                    collide_f(std::true_type{});
                else
                    collide_f(std::false_type{});
                // Eq. BGK-NS with Eqs. G_i, GGi.  Per direction pair: even part
                // E = w [itg A + c.u (4.5 rho itg c.u + 3 k drho c.grad phi)], odd part
                // O = w [3 rho itg c.u + 3 k c.F], k = 1 - itg/2, A = 3p - 1.5 rho |u|^2;
                // coefficients at w = 1/9, the diagonals take a quarter at the end
                const double A = fma(-1.5, ruu, p3);
                const double omg = 1.0 - itg;
                const double it9 = (1.0 / 9.0) * itg, k9 = fma(-0.5, it9, 1.0 / 9.0);
                const double e0 = it9 * A, ri = rho * it9, e1 = 4.5 * ri, o1 = 3.0 * ri;
                const double e2 = (1.5 * P.drho) * k9, o2 = 3.0 * k9;
                auto pair = [&](double cu, double cF, double cq, double &s, double &d) {
                    const double E = fma(cu, fma(e2, cq, e1 * cu), e0);
                    const double O = fma(o2, cF, o1 * cu);
                    s = E + O;
                    d = E - O;
                };
                double s, d;
                gd[n] = relax64<INCG>(gv[0], itg, omg, itg * fma(4.0 / 9.0, A, -p3));
                pair(ux, Fx, qx, s, d);
                gd[2 * N + n] = relax64<INCG>(gv[2], itg, omg, s);
                gd[4 * N + n] = relax64<INCG>(gv[4], itg, omg, d);
                pair(uy, Fy, qy, s, d);
                gd[3 * N + n] = relax64<INCG>(gv[3], itg, omg, s);
                gd[1 * N + n] = relax64<INCG>(gv[1], itg, omg, d);
                pair(ux + uy, Fx + Fy, qx + qy, s, d);
                gd[5 * N + n] = relax64<INCG>(gv[5], itg, omg, 0.25 * s);
                gd[7 * N + n] = relax64<INCG>(gv[7], itg, omg, 0.25 * d);
                pair(uy - ux, Fy - Fx, qy - qx, s, d);
                gd[6 * N + n] = relax64<INCG>(gv[6], itg, omg, 0.25 * s);
                gd[8 * N + n] = relax64<INCG>(gv[8], itg, omg, 0.25 * d);
            }
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) fcur[i] = fnext[i];
        scur = snext;
    }

    if (PASS & PASS_DIAG) {
        __syncthreads();  // every flag write of the march is done
        double d_phi = dacc[0][lin], d_E = dacc[1][lin],
               d_bud = 1.5 * dacc[2][lin] - 0.5 * dacc[3][lin];
        double d_u2 = facc[0][lin], d_mumin = facc[1][lin], d_mumax = facc[2][lin],
               d_bad = sm.bad ? 1.0 : 0.0;
        write_partial<NW>(sm.red, lin, d_phi, d_E, d_u2, d_mumin, d_mumax, d_bud, d_bad,
                          a.partials + part);
    }
}

// The FP64 time step of a grid too small to fill the chip.  A warp takes 64
// cycles for any FP64 instruction, whatever its active lanes, and each of the
// SM's four schedulers has one such pipe; with fewer warps than pipes the step
// takes the operations of one warp, one after the other (7.2 us for the 180 of
// two rows of d2q9_tile64).  Here a tile of 16 x 2 nodes is one CTA of four
// warps, one per scheduler, that share the node update: every warp holds the 32
// nodes and does a part of their operations, so that about 85 of them are in
// sequence.  Each value is formed by the expressions of d2q9_tile64.  16 x 128:
// 9.5 -> 4.9 us per step.
//   1  phi of the tile and two halo rows and columns (one node per thread)
//   2  v, d of one halo row                 warp 3: rho u's sum, sum of g
//   3  mu of one halo row and column          (while 1 .. 3 run elsewhere)
//   4  warp 0: F    warp 1: rho, 1/rho, 1/tau_g and what follows from them
//      warp 2: 2 grad(phi)
//   5  warp 0: f and S     warp 1: g along the axes
//      warp 2, 3: g along one diagonal each, warp 3 the rest population
constexpr int SM64_TX = 16, SM64_NT = 128;
struct SmallSmem64 {
    static constexpr int WP = SM64_TX + 4, WM = SM64_TX + 2;
    double phs[6 * WP], vs[4 * WP], ds[4 * WP], mus[4 * WM];
    double snz[32];               // sum of the moving f of the tile's nodes
    double w[14][32];             // stage 2 .. 4 results per node
};
template <bool INCG>
__global__ void __launch_bounds__(SM64_NT, 4)
    d2q9_small64_kernel(const StepParams<double> P, PassArgs a)
{
    constexpr int TX = SM64_TX, WP = SmallSmem64::WP, WM = SmallSmem64::WM;
    __shared__ SmallSmem64 sm;
    const int bx = pdl_wait(blockIdx.x);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = P.nx, ny = P.ny;
    const unsigned N = (unsigned)P.N;
    const int x0 = bx * TX, y0 = blockIdx.y * 2;
    const double *__restrict__ fsrc = static_cast<const double *>(a.f_src);
    const double *__restrict__ gsrc = static_cast<const double *>(a.g_src);
    // this thread's node in stages 2 .. 5
    const int tx = lane & 15, ty = lane >> 4;
    const int xo = x0 + tx, yo = y0 + ty;
    const bool ok = xo < nx && yo < ny;
    const unsigned xO = wrapi(xo, nx), xOm = wrapi(xo - 1, nx), xOp = wrapi(xo + 1, nx);
    const unsigned rm = (unsigned)wrapi(yo - 1, ny) * nx, r0 = (unsigned)wrapi(yo, ny) * nx,
                   rp = (unsigned)wrapi(yo + 1, ny) * nx;
    const unsigned n = r0 + xO;
    double v[9], Sprev = 0.0;  // warp 0: the node's f; else its g
    pull9<true>(warp == 0 ? fsrc : gsrc, N, rm, r0, rp, xOm, xO, xOp, v);
    if (warp == 0) Sprev = __ldcs(static_cast<const double *>(a.S) + n);

    if (tid < 6 * WP) {  // stage 1: ring rows y0 - 2 .. y0 + 3, columns x0 - 2 .. x0 + 17
        const int r = tid / WP, c = tid - r * WP;
        const int xx = x0 - 2 + c, yy = y0 - 2 + r;
        const unsigned q0 = (unsigned)wrapi(yy, ny) * nx, qm = (unsigned)wrapi(yy - 1, ny) * nx,
                       qp = (unsigned)wrapi(yy + 1, ny) * nx;
        double h[9];
        pull9<true>(fsrc, N, qm, q0, qp, (unsigned)wrapi(xx - 1, nx), (unsigned)wrapi(xx, nx),
                    (unsigned)wrapi(xx + 1, nx), h);
        const double s = sum_moving(h);
        sm.phs[tid] = h[0] + s;
        if (r >= 2 && r < 4 && c >= 2 && c < TX + 2) sm.snz[(r - 2) * 16 + c - 2] = s;
    }
    __syncthreads();
    if (tid < 4 * WP) {  // stage 2: rows y0 - 1 .. y0 + 2 (ring rows 1 .. 4)
        const double c = sm.phs[tid + WP], nn = sm.phs[tid + 2 * WP], ss = sm.phs[tid];
        sm.vs[tid] = (nn - c) + (ss - c);
        sm.ds[tid] = nn - ss;
    }
    if (warp == 3) {
        const double ga = v[5] - v[7], gb = v[8] - v[6];
        sm.w[0][lane] = (v[2] - v[4]) + (ga + gb);
        sm.w[1][lane] = (v[3] - v[1]) + (ga - gb);
        sm.w[2][lane] = sum_moving(v);
    }
    // (warp 3 joins the barrier of stage 2 late; stage 3 is 72 nodes of warps 0 .. 2)
    __syncthreads();
    if (tid < 4 * WM) {  // stage 3: the same rows, columns x0 - 1 .. x0 + 16
        const int r = tid / WM, j = tid - r * WM + 1;
        const double *p0 = sm.phs + (r + 1) * WP, *vr = sm.vs + r * WP;
        const double c = p0[j];
        const double h = (p0[j + 1] - c) + (p0[j - 1] - c);
        double mu = 4.0 * P.beta * (c - P.phil) * (c - P.phiv) * (c - P.phibar);
        mu = fma(-P.kappa, h, mu);
        mu = fma(-(P.kappa * (2.0 / 3.0)), vr[j], mu);
        sm.mus[tid] = fma(-(P.kappa * (1.0 / 6.0)), vr[j + 1] + vr[j - 1], mu);
    }
    __syncthreads();
    const int j = tx + 2, k = tx + 1;
    const double *p0 = sm.phs + (ty + 2) * WP, *vr = sm.vs + (ty + 1) * WP,
                 *dr = sm.ds + (ty + 1) * WP;
    const double *mm = sm.mus + ty * WM, *m0 = mm + WM, *mp = m0 + WM;
    const double phi = p0[j];
    if (warp == 0) {  // stage 4
        const double da = mp[k + 1] - mm[k - 1], db = mm[k + 1] - mp[k - 1];
        const double f3 = (-1.0 / 3.0) * phi;
        sm.w[3][lane] = fma(f3, fma(0.25, da + db, m0[k + 1] - m0[k - 1]), P.G[0]);
        sm.w[4][lane] = fma(f3, fma(0.25, da - db, mp[k] - mm[k]), P.G[1]);
    } else if (warp == 1) {
        const double dphi = phi - P.phiv;
        const double rho = fma(P.drho, dphi, P.rhov);
        const double taug = fma(3.0 * P.dnu, dphi, fma(3.0, P.nuv, 0.5));
        const double itg = rcp64(taug), it9 = (1.0 / 9.0) * itg, ri = rho * it9;
        const double k9 = fma(-0.5, it9, 1.0 / 9.0);
        sm.w[5][lane] = rho;
        sm.w[6][lane] = rcp64(rho);
        sm.w[7][lane] = itg;
        sm.w[8][lane] = it9;
        sm.w[9][lane] = ri;
        sm.w[10][lane] = k9;
    } else if (warp == 2) {
        sm.w[11][lane] = fma(1.0 / 6.0, vr[j + 1] - vr[j - 1], p0[j + 1] - p0[j - 1]);
        sm.w[12][lane] = fma(1.0 / 6.0, dr[j + 1] + dr[j - 1], (2.0 / 3.0) * dr[j]);
    }
    __syncthreads();
    if (!ok) return;
    // stage 5
    const double Fx = sm.w[3][lane], Fy = sm.w[4][lane], irho = sm.w[6][lane];
    const double qx = sm.w[11][lane], qy = sm.w[12][lane];
    const double ux = fma(0.5, Fx, sm.w[0][lane]) * irho, uy = fma(0.5, Fy, sm.w[1][lane]) * irho;
    const double S2 = fma(ux, qx, uy * qy);
    double *__restrict__ fd = static_cast<double *>(a.f_dst);
    double *__restrict__ gd = static_cast<double *>(a.g_dst);
    if (warp == 0) {
        static_cast<double *>(a.S_out)[n] = 0.5 * S2;
        const double Sh = fma(0.75, S2, -0.5 * Sprev);
        const double itf = P.inv_tauf, omf = 1.0 - itf;
        const double z = (itf * P.alpha) * m0[k];
        fd[n] = v[0] + fma(itf, sm.snz[lane], fma(-5.0 / 9.0, z, (-8.0 / 9.0) * Sh));
        const double ka = (1.0 / 9.0) * fma(-0.5, Sh, z), kd = (1.0 / 36.0) * (z + Sh);
        auto collide_f = [&](auto inc) {
#pragma unroll
            for (int i = 1; i < 9; ++i)
                fd[i * N + n] = relax64<inc.value>(v[i], itf, omf, i < 5 ? ka : kd);
        };
        if (P.incr & INCR_F)
            collide_f(std::true_type{});
        else
            collide_f(std::false_type{});
        return;
    }
    const double rho = sm.w[5][lane], itg = sm.w[7][lane], it9 = sm.w[8][lane],
                 ri = sm.w[9][lane], k9 = sm.w[10][lane];
    const double uu = fma(ux, ux, uy * uy), ruu = rho * uu;
    const double p3 = 1.8 * fma(-2.0 / 3.0, ruu, fma(0.25 * P.drho, S2, sm.w[2][lane]));
    const double A = fma(-1.5, ruu, p3), omg = 1.0 - itg;
    const double e0 = it9 * A, e1 = 4.5 * ri, o1 = 3.0 * ri;
    const double e2 = (1.5 * P.drho) * k9, o2 = 3.0 * k9;
    auto pair = [&](double cu, double cF, double cq, double &s, double &d) {
        const double E = fma(cu, fma(e2, cq, e1 * cu), e0);
        const double O = fma(o2, cF, o1 * cu);
        s = E + O;
        d = E - O;
    };
    double s, d;
    if (warp == 1) {
        pair(ux, Fx, qx, s, d);
        gd[2 * N + n] = relax64<INCG>(v[2], itg, omg, s);
        gd[4 * N + n] = relax64<INCG>(v[4], itg, omg, d);
        pair(uy, Fy, qy, s, d);
        gd[3 * N + n] = relax64<INCG>(v[3], itg, omg, s);
        gd[1 * N + n] = relax64<INCG>(v[1], itg, omg, d);
    } else if (warp == 2) {
        pair(ux + uy, Fx + Fy, qx + qy, s, d);
        gd[5 * N + n] = relax64<INCG>(v[5], itg, omg, 0.25 * s);
        gd[7 * N + n] = relax64<INCG>(v[7], itg, omg, 0.25 * d);
    } else {
        gd[n] = relax64<INCG>(v[0], itg, omg, itg * fma(4.0 / 9.0, A, -p3));
        pair(uy - ux, Fy - Fx, qy - qx, s, d);
        gd[6 * N + n] = relax64<INCG>(v[6], itg, omg, 0.25 * s);
        gd[8 * N + n] = relax64<INCG>(v[8], itg, omg, 0.25 * d);
    }
}
