// Two nodes adjacent in x per thread on the paired FP32 datapath: shared by the
// D3Q19 passes.  Internal header.
#pragma once

#include <cuda_runtime.h>

namespace wblbm {

// The paired FP32 datapath: two independent lanes per instruction, each
// rounding as the scalar instruction does.  The lanes are the thread's two
// nodes.
__device__ __forceinline__ float2 f2(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 add2(float2 x, float2 y) { return __fadd2_rn(x, y); }
__device__ __forceinline__ float2 mul2(float2 x, float2 y) { return __fmul2_rn(x, y); }
__device__ __forceinline__ float2 fma2(float2 x, float2 y, float2 z) { return __ffma2_rn(x, y, z); }
// x - y as one multiply-add by -1 (the same single rounding)
__device__ __forceinline__ float2 sub2(float2 x, float2 y) { return __ffma2_rn(y, f2(-1.0f), x); }
__device__ __forceinline__ float2 neg2(float2 x) { return __fmul2_rn(x, f2(-1.0f)); }
// sum_d c_d v_d of a velocity c (components 0, 1, -1; the first non-zero one may be -1)
__device__ __forceinline__ float2 dot_c(int cx, int cy, int cz, float2 x, float2 y, float2 z)
{
    float2 s = cx ? (cx > 0 ? x : neg2(x)) : (cy ? (cy > 0 ? y : neg2(y)) : (cz > 0 ? z : neg2(z)));
    if (cx && cy) s = cy > 0 ? add2(s, y) : sub2(s, y);
    if ((cx || cy) && cz) s = cz > 0 ? add2(s, z) : sub2(s, z);
    return s;
}
// the pair of floats at index c, c + 1 of a shared-memory plane (one 64-bit read where c is even)
__device__ __forceinline__ float2 pair_at(const float *pl, int c, bool even)
{
    if (even) return *reinterpret_cast<const float2 *>(pl + c);
    return make_float2(pl[c], pl[c + 1]);
}
// Eq. gradient on D3Q19 from the ring planes below (m), at (z) and above (p), rows SX apart,
// c even: (1/6) face differences + (1/12) edge differences
__device__ __forceinline__ void grad3_pair(const float *m, const float *z, const float *p, int c,
                                           int SX, float2 out[3])
{
    const float2 xe = pair_at(z, c + 1, false), xw = pair_at(z, c - 1, false);
    const float2 yn = pair_at(z, c + SX, true), ys = pair_at(z, c - SX, true);
    const float2 pc = pair_at(p, c, true), mc = pair_at(m, c, true);
    const float2 ne = pair_at(z, c + SX + 1, false), nw = pair_at(z, c + SX - 1, false);
    const float2 se = pair_at(z, c - SX + 1, false), sw = pair_at(z, c - SX - 1, false);
    const float2 pe = pair_at(p, c + 1, false), pw = pair_at(p, c - 1, false);
    const float2 me = pair_at(m, c + 1, false), mw = pair_at(m, c - 1, false);
    const float2 pn = pair_at(p, c + SX, true), ps = pair_at(p, c - SX, true);
    const float2 mn = pair_at(m, c + SX, true), ms = pair_at(m, c - SX, true);
    const float2 k6 = f2(1.0f / 6.0f), k12 = f2(1.0f / 12.0f);
    out[0] = fma2(k6, sub2(xe, xw),
                  mul2(k12, add2(add2(add2(sub2(ne, nw), sub2(se, sw)), sub2(pe, pw)),
                                 sub2(me, mw))));
    out[1] = fma2(k6, sub2(yn, ys),
                  mul2(k12, add2(add2(add2(sub2(ne, se), sub2(nw, sw)), sub2(pn, ps)),
                                 sub2(mn, ms))));
    out[2] = fma2(k6, sub2(pc, mc),
                  mul2(k12, add2(add2(add2(sub2(pe, me), sub2(pw, mw)), sub2(pn, mn)),
                                 sub2(ps, ms))));
}

}  // namespace wblbm
