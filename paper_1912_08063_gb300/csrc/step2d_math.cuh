// Arithmetic of one 2-D step on a group of 4 points (shared by every 2-D step kernel, so
// all of them give the same results bit for bit): the order-2M Laplacian from an x-window
// and z-sums, and the damped leapfrog update.
#pragma once

#include <cuda_runtime.h>

#include "fwi_internal.h"

namespace fwi {
namespace s2d {

__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// Adds the z-neighbours at distance k of a group, rows lo and hi, to its z-sums (za: points
// 0, 1; zb: points 2, 3).  Every kernel calls it for k = 1 .. M in this order.
__device__ __forceinline__ void z_pair(float ck, float4 up, float4 dn, float2 &za, float2 &zb)
{
    const float2 cc = make_float2(ck, ck);
    za = __ffma2_rn(cc, __fadd2_rn(lo2(dn), lo2(up)), za);
    zb = __ffma2_rn(cc, __fadd2_rn(hi2(dn), hi2(up)), zb);
}

// L c at the 4 points of a group from its z-sums and its x-window w (groups x0 - M .. x0 +
// 3 + M, the centre group c at w[M .. M + 3]).  x-sums: odd and even offsets in two chains
// per point; packed, even offsets pair points (0, 1) and (2, 3) on aligned register pairs
// and odd ones (1, 2), with points 0 and 3 alone.
template <int M>
__device__ __forceinline__ void lap_x(const float (&w)[4 + 2 * M], float4 c, const Coefs &cf,
                                      float2 za, float2 zb, float2 &l0, float2 &l1)
{
    const float2 zero = make_float2(0.f, 0.f);
    float2 ea = zero, eb = zero, om = zero;   // even: points (0, 1), (2, 3); odd: (1, 2)
    float o0 = 0.0f, o3 = 0.0f;               // odd: points 0 and 3
#pragma unroll
    for (int k = 1; k <= M; ++k) {
        const float ck = cf.cx[k];
        const float2 ck2 = make_float2(ck, ck);
        if ((k & 1) == 0) {
            ea = __ffma2_rn(ck2, __fadd2_rn(make_float2(w[M + k], w[M + k + 1]),
                                            make_float2(w[M - k], w[M - k + 1])), ea);
            eb = __ffma2_rn(ck2, __fadd2_rn(make_float2(w[M + 2 + k], w[M + 3 + k]),
                                            make_float2(w[M + 2 - k], w[M + 3 - k])), eb);
        } else {
            om = __ffma2_rn(ck2, __fadd2_rn(make_float2(w[M + 1 + k], w[M + 2 + k]),
                                            make_float2(w[M + 1 - k], w[M + 2 - k])), om);
            o0 = fmaf(ck, w[M + k] + w[M - k], o0);
            o3 = fmaf(ck, w[M + 3 + k] + w[M + 3 - k], o3);
        }
    }
    const float2 c0 = make_float2(cf.c0, cf.c0);
    l0 = __ffma2_rn(c0, lo2(c), __fadd2_rn(za, __fadd2_rn(make_float2(o0, om.x), ea)));
    l1 = __ffma2_rn(c0, hi2(c), __fadd2_rn(zb, __fadd2_rn(make_float2(om.y, o3), eb)));
}

// The z-sums of RZ consecutive rows of a group from a column of rows in shared memory (row i
// at col + i * stride, output row r at row r + M), loaded outwards so that only the rows
// between the nearest and the farthest in use are held; c[r] receives the centre rows.
template <int M, int RZ>
__device__ __forceinline__ void z_block(const float *col, int stride, const Coefs &cf, float4 (&c)[RZ],
                                        float2 (&za)[RZ], float2 (&zb)[RZ])
{
    float4 q[RZ + 2 * M];
#pragma unroll
    for (int r = 0; r < RZ; ++r) {
        c[r] = q[M + r] = *(const float4 *)(col + (M + r) * stride);
        za[r] = zb[r] = make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int k = 1; k <= M; ++k) {
        q[M - k] = *(const float4 *)(col + (M - k) * stride);
        q[M + RZ - 1 + k] = *(const float4 *)(col + (M + RZ - 1 + k) * stride);
#pragma unroll
        for (int r = 0; r < RZ; ++r) z_pair(cf.cz[k], q[M + r - k], q[M + r + k], za[r], zb[r]);
    }
}

// Approximate reciprocal of the damping factor 1 + s, a normal number near 1: rcp.approx.ftz is
// within 1 ulp of the exact one (PTX ISA).
__device__ __forceinline__ float rcp_damp(float d)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return r;
}

// The damped update of a group: (2c + W lap - (1 - s) prev [+ srcv at point se]) / (1 + s),
// packed; the quotient is the product with the approximate reciprocal of 1 + s.
__device__ __forceinline__ float4 update4(float4 c, float2 l0, float2 l1, float4 pv, float4 Wv,
                                          float4 sx, float sz, int se, float srcv)
{
    const float2 two = make_float2(2.0f, 2.0f), one = make_float2(1.0f, 1.0f), m1 = make_float2(-1.0f, -1.0f);
    const float2 s2 = make_float2(sz, sz);
    const float2 sa = __fadd2_rn(lo2(sx), s2), sb = __fadd2_rn(hi2(sx), s2);
    float2 a = __ffma2_rn(__fadd2_rn(sa, m1), lo2(pv), __ffma2_rn(lo2(Wv), l0, __fmul2_rn(two, lo2(c))));
    float2 b = __ffma2_rn(__fadd2_rn(sb, m1), hi2(pv), __ffma2_rn(hi2(Wv), l1, __fmul2_rn(two, hi2(c))));
    if (se >= 0) {
        if (se == 0) a.x += srcv;
        else if (se == 1) a.y += srcv;
        else if (se == 2) b.x += srcv;
        else b.y += srcv;
    }
    const float2 da = __fadd2_rn(one, sa), db = __fadd2_rn(one, sb);
    a = __fmul2_rn(a, make_float2(rcp_damp(da.x), rcp_damp(da.y)));
    b = __fmul2_rn(b, make_float2(rcp_damp(db.x), rcp_damp(db.y)));
    return make_float4(a.x, a.y, b.x, b.y);
}

}  // namespace s2d
}  // namespace fwi
