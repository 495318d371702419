// 3-D time step on GB300 (sm_103a) for grids that stay in L2: one brick per CTA, no streaming.
//
// The streaming kernels (k_step3d_tm.cuh, k_step3d.cuh) walk a tile column plane by plane so
// that each plane is read from DRAM once.  On a grid of a few million points that leaves most
// SMs with one CTA, or none, walking some 50 planes one after the other, 2M of them warm-up,
// while every field sits in L2 anyway.  Here a CTA owns a brick of 32 x 8 x 4 points and asks
// for everything at once: the brick with its x- and y-halo as one TMA box [z][y][x], the M
// planes below and above it (without corners) as two more, and the pointwise operands (prev,
// W; u^m and g in kModeAdj) straight into registers.  A warp owns two planes of the brick, a
// thread 4 x 2 x 2 points (radius 4's reverse mode: one plane, 4 x 2 x 1).  The halo re-reads
// (8.5 floats a point at radius 8, 4.5 at radius 4) go to L2, not to DRAM, and there is one
// wait per CTA instead of one per plane.
//
// The sums run in the order of the streaming kernel that takes the same radius and mode
// otherwise, so both give the same results bit for bit.
//
// Measured on GB300 against the streaming kernels, us per launch with about 4 us of event
// overhead, forward / forward + store / reverse (computed cubes, 40 cells wider than named):
//   radius 4:   56^3  14.0 / 14.6 / 13.3 ->  8.9 /  9.6 / 10.2   96^3  18.6 / 20.6 / 22.4 -> 14.5 / 16.8 / 20.2
//              120^3  20.0 / 21.6 / 24.5 -> 16.5 / 19.1 / 26.1  160^3  32.9 / 38.7 / 49.8 -> 38.1 / 45.4 / 61.7
//   radius 8:   56^3  18.7 / 20.7 / 24.2 -> 10.5 / 10.8 / 10.6   96^3  27.0 / 29.0 / 31.3 -> 17.1 / 20.4 / 23.1
//              120^3  28.5 / 30.7 / 32.3 -> 21.3 / 24.9 / 27.4  160^3  46.0 / 51.0 / 55.6 -> 45.9 / 57.8 / 66.5
// (before the streaming plans of step3d.h cut columns into equal parts the radius-8 streaming
// steps took 45.5 / 49.2 / 63.0 at 96^3).  What bounds it at 96^3 is latency: issue slots 35 %
// busy with 11 warps an SM, the warps waiting on global loads and shared memory.
// Brick: 32 x 8 x 8 by four warps (96^3 radius 8 18.8 / 20.4 / 25.5, 160^3 46.5 / 52.0 / 74.4),
// 32 x 16 x 8 (19.6 / 21.0 / 28.4, 52.0 / 56.4 / 91.9), 32 x 8 x 16 (19.7 / 21.1 / 28.4, 50.7 /
// 55.5 / 93.6) read fewer halo floats but leave fewer, larger CTAs and were no faster; one
// plane per warp everywhere 18.7 / 20.3 / 24.3, 49.4 / 53.7 / 71.6.  The halo without its corners (a box
// of the brick's columns and one for each side: 12 % fewer bytes, seven CTAs an SM instead of
// six) was slower too: 18.4 / 22.4 / 24.5 at 96^3, 21.6 / 26.8 / 28.8 at 120^3.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>

#include "k_step3d.cuh"
#include "pdl.cuh"
#include "taps.cuh"

namespace fwi {
namespace {

using s3d::absmax_nan;
using s3d::hi2;
using s3d::lo2;
using s3d::mbar_expect_tx;
using s3d::mbar_init;
using s3d::mbar_wait;
using s3d::rcp_fast;
using s3d::smem_u32;
using s3d::src_image;
using s3d::taylor;
using s3d::taylor_centre3;
using s3d::tma_load4;

template <int M_, int MODE, bool ISO_>
struct Brick {
    static constexpr int M = M_;
    static constexpr bool ISO = ISO_;
    static constexpr int TX = 32, TY = 8, TZ = 4, RY = 2;

    static constexpr int SX = TX + 2 * M, SY = TY + 2 * M;
    static constexpr int MID = SX * SY * TZ, ARM = TX * TY * M;   // floats
    static constexpr int SMEM = (MID + 2 * ARM) * 4 + 128;
    // radius 4's reverse mode sums in the register-queue kernel's order
    static constexpr bool QUEUE = M == 4 && MODE == kModeAdj;
    static constexpr int RZ = QUEUE ? 1 : 2;                      // planes per warp
    static constexpr int NT = 32 * TZ / RZ;
    static constexpr int MINB = QUEUE ? 4 : MODE == kModeAdj ? 6 : 8;
};

template <class C>
__device__ __forceinline__ float wx(const Step3dParams &p, int k) { return C::ISO ? taylor<C::M>(k) : p.cx[k]; }
template <class C>
__device__ __forceinline__ float wy(const Step3dParams &p, int k) { return C::ISO ? taylor<C::M>(k) : p.cy[k]; }
template <class C>
__device__ __forceinline__ float wz(const Step3dParams &p, int k) { return C::ISO ? taylor<C::M>(k) : p.cz[k]; }

__device__ __forceinline__ void fma4(float2 &a, float2 &b, float c, float4 v)
{
    const float2 c2 = make_float2(c, c);
    a = __ffma2_rn(c2, lo2(v), a);
    b = __ffma2_rn(c2, hi2(v), b);
}

// The x- and y-parts of the Laplacian of one plane (hk: its tile with halo) at this thread's
// two rows, and the rows' values.  SEMI order: (y + even x) + odd x, then the centre term;
// QUEUE order returns y- and x-sums apart (ys, lx).
template <class C>
__device__ __forceinline__ void plane_xy(const Step3dParams &p, const float *hk, float4 (&ctr)[C::RY],
                                         float2 (&a)[C::RY][2], float2 (&lx)[C::RY][2])
{
    constexpr int M = C::M, SX = C::SX, RY = C::RY;
    float2 ya[RY][2], yb[RY][2];
#pragma unroll
    for (int r = 0; r < RY; ++r) ya[r][0] = ya[r][1] = yb[r][0] = yb[r][1] = make_float2(0.f, 0.f);
#pragma unroll
    for (int t = 0; t < 2 * M + RY; ++t) {
        const float4 v = *(const float4 *)(hk + t * SX + M);
#pragma unroll
        for (int r = 0; r < RY; ++r) {
            const int d = t - M - r;
            if (d == 0) ctr[r] = v;
            else if (d >= -M && d <= M) {
                const float c = wy<C>(p, d < 0 ? -d : d);
                if (t & 1) fma4(ya[r][0], ya[r][1], c, v);
                else fma4(yb[r][0], yb[r][1], c, v);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RY; ++r) {
        float w[4 + 2 * M];
        const float *row = hk + (r + M) * SX;
#pragma unroll
        for (int g = 0; g < (4 + 2 * M) / 4; ++g) {
            const float4 v = g == M / 4 ? ctr[r] : *(const float4 *)(row + 4 * g);
            w[4 * g] = v.x, w[4 * g + 1] = v.y, w[4 * g + 2] = v.z, w[4 * g + 3] = v.w;
        }
        // even offsets pair points (0, 1) and (2, 3), odd ones (1, 2), 0 and 3 alone
        const float2 zero = make_float2(0.f, 0.f);
        float2 ea = C::QUEUE ? zero : ya[r][0], eb = C::QUEUE ? zero : ya[r][1], xm = zero;
        float x0 = 0.0f, x3 = 0.0f;
#pragma unroll
        for (int k = 1; k <= M; ++k) {
            const float ck = wx<C>(p, k);
            const float2 ck2 = make_float2(ck, ck);
            if ((k & 1) == 0) {
                ea = __ffma2_rn(ck2, __fadd2_rn(make_float2(w[M + k], w[M + k + 1]),
                                                make_float2(w[M - k], w[M - k + 1])), ea);
                eb = __ffma2_rn(ck2, __fadd2_rn(make_float2(w[M + 2 + k], w[M + 3 + k]),
                                                make_float2(w[M + 2 - k], w[M + 3 - k])), eb);
            } else {
                xm = __ffma2_rn(ck2, __fadd2_rn(make_float2(w[M + 1 + k], w[M + 2 + k]),
                                                make_float2(w[M + 1 - k], w[M + 2 - k])), xm);
                x0 = fmaf(ck, w[M + k] + w[M - k], x0);
                x3 = fmaf(ck, w[M + 3 + k] + w[M + 3 - k], x3);
            }
        }
        if (C::QUEUE) {
            a[r][0] = __fadd2_rn(ya[r][0], yb[r][0]);
            a[r][1] = __fadd2_rn(ya[r][1], yb[r][1]);
            lx[r][0] = __fadd2_rn(make_float2(x0, xm.x), ea);
            lx[r][1] = __fadd2_rn(make_float2(xm.y, x3), eb);
        } else {
            const float2 c0 = C::ISO ? make_float2(taylor_centre3<M>(), taylor_centre3<M>()) : p.c02;
            a[r][0] = __ffma2_rn(c0, lo2(ctr[r]),
                                 __fadd2_rn(__fadd2_rn(ea, yb[r][0]), make_float2(x0, xm.x)));
            a[r][1] = __ffma2_rn(c0, hi2(ctr[r]),
                                 __fadd2_rn(__fadd2_rn(eb, yb[r][1]), make_float2(xm.y, x3)));
        }
    }
}

// TAPS: an off-grid source is added too (an instantiation of its own).
template <int M, int MODE, bool ISO, bool TAPS>
__global__ void __launch_bounds__(Brick<M, MODE, ISO>::NT, Brick<M, MODE, ISO>::MINB)
k_step3d_brick(const __grid_constant__ Step3dParams p, const __grid_constant__ CUtensorMap map_mid,
               const __grid_constant__ CUtensorMap map_arm, int tiles_z)
{
    using C = Brick<M, MODE, ISO>;
    constexpr int TX = C::TX, TY = C::TY, TZ = C::TZ, RY = C::RY, RZ = C::RZ, SX = C::SX, SY = C::SY;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float *mid = (float *)smem, *zlo = mid + C::MID, *zhi = zlo + C::ARM;
    __shared__ __align__(8) uint64_t bar;
    const int tid = threadIdx.x, tx = tid & 7, ty = (tid >> 3) & 3, tz = tid >> 5;
    const int shot = blockIdx.z / tiles_z, bz = blockIdx.z - shot * tiles_z;
    const int X0 = blockIdx.x * TX, Y0 = blockIdx.y * TY, Z0 = bz * TZ;
    pdl_next();
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    const int x0 = X0 + 4 * tx, y0 = Y0 + RY * ty, zb = Z0 + RZ * tz;
    const int px = p.px;
    const int64_t off = (int64_t)zb * p.plane + (int64_t)y0 * px + x0;
    const int64_t sb = (int64_t)shot * p.field + off;
    float *out = p.out + sb;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    bool ok[RZ][RY];
    float4 pv[RZ][RY], Wv[RZ][RY], gv[MODE == kModeAdj ? RZ : 1][RY];
    uint4 ur[MODE == kModeAdj ? RZ : 1][RY];
    const int afmt = p.aux_fmt;
#pragma unroll
    for (int i = 0; i < RZ; ++i)
#pragma unroll
        for (int r = 0; r < RY; ++r) {
            ok[i][r] = x0 < p.nx && y0 + r < p.ny && zb + i < p.nz;
            Wv[i][r] = ok[i][r] ? __ldg((const float4 *)(p.W + off + (int64_t)i * p.plane + r * px)) : zero4;
        }
    const float4 sx = x0 < p.nx ? __ldg((const float4 *)(p.sig_x + x0)) : zero4;   // padded with zeros
    float syr[RY], szr[RZ];
#pragma unroll
    for (int r = 0; r < RY; ++r) syr[r] = y0 + r < p.ny ? p.sig_y[y0 + r] : 0.0f;
#pragma unroll
    for (int i = 0; i < RZ; ++i) szr[i] = zb + i < p.nz ? p.sig_z[zb + i] : 0.0f;
    pdl_wait();
    if (tid == 0) {
        mbar_expect_tx(&bar, (C::MID + 2 * C::ARM) * 4);
        tma_load4(mid, &map_mid, X0 - M, Y0 - M, Z0, shot, &bar);
        tma_load4(zlo, &map_arm, X0, Y0, Z0 - M, shot, &bar);
        tma_load4(zhi, &map_arm, X0, Y0, Z0 + TZ, shot, &bar);
    }
#pragma unroll
    for (int i = 0; i < RZ; ++i)
#pragma unroll
        for (int r = 0; r < RY; ++r) {
            const int64_t o = (int64_t)i * p.plane + r * px;
            pv[i][r] = ok[i][r] ? *(const float4 *)(out + o) : zero4;
            if (MODE == kModeAdj) {
                gv[i][r] = ok[i][r] ? *(const float4 *)(p.g + sb + o) : zero4;
                const int64_t uo = (int64_t)shot * p.aux_stride + off + o;
                ur[i][r] = make_uint4(0u, 0u, 0u, 0u);
                // past L1 (96^3 gradient 20.42 ms; through L1 20.47, and 20.69 with the two
                // formats in one branch)
                if (ok[i][r] && afmt == 0) ur[i][r] = load_cg((const uint4 *)((const float *)p.aux + uo));
                if (ok[i][r] && afmt != 0) {
                    const uint2 h = load_cg((const uint2 *)((const unsigned short *)p.aux + uo));
                    ur[i][r].x = h.x;
                    ur[i][r].y = h.y;
                }
            }
        }
    const int n = (p.n_dev ? *p.n_dev : 0) + p.n;
    int src_i = -1, src_r = 0, src_e = 0;
    float srcv = 0.0f;
    if (p.src_off) {
        const int64_t s = p.src_off[shot];
        const int sz = (int)(s / p.plane), rem = (int)(s - (int64_t)sz * p.plane);
        const int sy = rem / px, sxx = rem - sy * px;
        if (sz >= zb && sz < zb + RZ && sy >= y0 && sy < y0 + RY && sxx >= x0 && sxx < x0 + 4) {
            src_i = sz - zb;
            src_r = sy - y0;
            src_e = sxx - x0;
            srcv = p.dt2 * p.wavelet[(int64_t)shot * p.nt + n];
        }
    }
    bool taps = false;   // an off-grid source's taps meet this thread's block
    if (TAPS) {
        taps = taps_meet(p.src_pts[shot], 3, zb, RZ, y0, RY, x0);
        if (taps) srcv = p.dt2 * p.wavelet[(int64_t)shot * p.nt + n];
    }
    float sca = 1.0f, scd = 1.0f;
    if (MODE == kModeStepStore) {
        const float2 sc = store_scales(p.st_max, shot, p.st_dtype);
        sca = sc.x;
        scd = sc.y;
    }
    const float ainv = (MODE == kModeAdj && p.aux_scale) ? 1.0f / p.aux_scale[2 * shot] : 1.0f;
    if (MODE != kModeAdj && tid == 0 && blockIdx.x == 0 && blockIdx.y == 0 && bz == 0)
        store_bookkeeping(p.st_max, shot, p.st_dtype, p.st_scale, p.err, p.max_clear);
    __syncthreads();   // the barrier is initialised
    if (!mbar_wait(&bar, 0)) {
        // a bounded wait gave up: report, then give the copies a bounded chance to land
        // before the CTA's shared memory is released
        if (tid == 0) atomicOr(p.err, 2u);
        (void)mbar_wait(&bar, 0);
        return;
    }

    // plane Z0 + zz of this thread's columns, rows 0 and 1 (zz uniform per warp)
    auto rows_of = [&](int zz, float4 (&v)[RY]) {
        const float *q;
        int stride;
        if (zz < 0 || zz >= TZ) {
            q = (zz < 0 ? zlo + (zz + M) * (TX * TY) : zhi + (zz - TZ) * (TX * TY)) + RY * ty * TX + 4 * tx;
            stride = TX;
        } else {
            q = mid + zz * (SX * SY) + (RY * ty + M) * SX + 4 * tx + M;
            stride = SX;
        }
#pragma unroll
        for (int r = 0; r < RY; ++r) v[r] = *(const float4 *)(q + r * stride);
    };
    // q[M + d]: rows of plane zb + d, d = -M .. RZ - 1 + M
    float4 q[2 * M + RZ][RY];
    float2 acc[RZ][RY][2], lx[RZ][RY][2];
    const int zt = RZ * tz;
#pragma unroll
    for (int i = 0; i < RZ; ++i)
        plane_xy<C>(p, mid + (zt + i) * (SX * SY) + RY * ty * SX + 4 * tx, q[M + i], acc[i], lx[i]);
    if (C::QUEUE) {
        float2 za[RZ][RY][2], zc[RZ][RY][2];   // odd and even distances
#pragma unroll
        for (int i = 0; i < RZ; ++i)
#pragma unroll
            for (int r = 0; r < RY; ++r)
                za[i][r][0] = za[i][r][1] = zc[i][r][0] = zc[i][r][1] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 1; k <= M; ++k) {
            rows_of(zt - k, q[M - k]);
            rows_of(zt + RZ - 1 + k, q[M + RZ - 1 + k]);
            const float c = wz<C>(p, k);
            const float2 cc = make_float2(c, c);
#pragma unroll
            for (int i = 0; i < RZ; ++i)
#pragma unroll
                for (int r = 0; r < RY; ++r) {
                    const float4 u = q[M + i + k][r], d = q[M + i - k][r];
                    float2(&z)[2] = (k & 1) ? za[i][r] : zc[i][r];
                    z[0] = __ffma2_rn(cc, __fadd2_rn(lo2(u), lo2(d)), z[0]);
                    z[1] = __ffma2_rn(cc, __fadd2_rn(hi2(u), hi2(d)), z[1]);
                }
        }
        const float2 c0 = C::ISO ? make_float2(taylor_centre3<M>(), taylor_centre3<M>()) : p.c02;
#pragma unroll
        for (int i = 0; i < RZ; ++i)
#pragma unroll
            for (int r = 0; r < RY; ++r) {
                const float4 c = q[M + i][r];
                const float2 s0 = __fadd2_rn(__fadd2_rn(za[i][r][0], zc[i][r][0]), acc[i][r][0]);
                const float2 s1 = __fadd2_rn(__fadd2_rn(za[i][r][1], zc[i][r][1]), acc[i][r][1]);
                acc[i][r][0] = __ffma2_rn(c0, lo2(c), __fadd2_rn(s0, lx[i][r][0]));
                acc[i][r][1] = __ffma2_rn(c0, hi2(c), __fadd2_rn(s1, lx[i][r][1]));
            }
    } else {
        // the planes below, nearest first; then the planes above, farthest first
#pragma unroll
        for (int m = 1; m <= M; ++m) {
            rows_of(zt - m, q[M - m]);
#pragma unroll
            for (int i = 0; i < RZ; ++i)
#pragma unroll
                for (int r = 0; r < RY; ++r) fma4(acc[i][r][0], acc[i][r][1], wz<C>(p, m), q[M + i - m][r]);
        }
#pragma unroll
        for (int k = M; k >= 1; --k) {
            if (k == M) {
#pragma unroll
                for (int i = 1; i < RZ; ++i) rows_of(zt + i + M, q[M + i + M]);
            }
            if (k >= RZ) rows_of(zt + k, q[M + k]);
#pragma unroll
            for (int i = 0; i < RZ; ++i)
#pragma unroll
                for (int r = 0; r < RY; ++r) fma4(acc[i][r][0], acc[i][r][1], wz<C>(p, k), q[M + i + k][r]);
        }
    }

    float mxa = 0.0f, mxd = 0.0f;
#pragma unroll
    for (int i = 0; i < RZ; ++i)
#pragma unroll
        for (int r = 0; r < RY; ++r) {
            const int z = zb + i, y = y0 + r;
            const int64_t o = (int64_t)i * p.plane + r * px;
            const float4 c = q[M + i][r], A = pv[i][r], B = Wv[i][r];
            float2 l0 = acc[i][r][0], l1 = acc[i][r][1];
            if (C::ISO) {
                const float2 ih = make_float2(p.inv_h2, p.inv_h2);
                l0 = __fmul2_rn(l0, ih);
                l1 = __fmul2_rn(l1, ih);
            }
            // prev + (2 (c - prev) + W lap [+ dt^2 w at the source]) / (1 + s)
            const float2 m1 = make_float2(-1.0f, -1.0f), two = make_float2(2.0f, 2.0f);
            const float2 dc0 = __ffma2_rn(lo2(A), m1, lo2(c)), dc1 = __ffma2_rn(hi2(A), m1, hi2(c));
            float2 t0 = __ffma2_rn(lo2(B), l0, __fmul2_rn(two, dc0));
            float2 t1 = __ffma2_rn(hi2(B), l1, __fmul2_rn(two, dc1));
            const bool at_src = i == src_i && r == src_r;
            if (MODE != kModeAdj && at_src) {
                if (src_e == 0) t0.x += srcv;
                else if (src_e == 1) t0.y += srcv;
                else if (src_e == 2) t1.x += srcv;
                else t1.y += srcv;
            }
            const float syz = syr[r] + szr[i];
            const float2 d0 = __fadd2_rn(make_float2(1.0f + sx.x, 1.0f + sx.y), make_float2(syz, syz));
            const float2 d1 = __fadd2_rn(make_float2(1.0f + sx.z, 1.0f + sx.w), make_float2(syz, syz));
            float2 o0 = __ffma2_rn(t0, make_float2(rcp_fast(d0.x), rcp_fast(d0.y)), lo2(A));
            float2 o1 = __ffma2_rn(t1, make_float2(rcp_fast(d1.x), rcp_fast(d1.y)), hi2(A));
            if (TAPS && taps && ok[i][r]) {
                float4 ov = make_float4(o0.x, o0.y, o1.x, o1.y);
                add_taps(p.src_pts[shot], 3, z, y, x0, srcv, szr[i] + syr[r], sx, ov);
                o0 = lo2(ov);
                o1 = hi2(ov);
            }
            if (p.rec_map && z == p.rec_z && ok[i][r]) {
                float ov[4] = {o0.x, o0.y, o1.x, o1.y};
                s3d::rec_epilogue<MODE>(p, shot, y, x0, n, ov);
                o0 = make_float2(ov[0], ov[1]);
                o1 = make_float2(ov[2], ov[3]);
            }
            if (MODE != kModeAdj && p.maxbits && ok[i][r]) {
                mxa = absmax_nan(absmax_nan(absmax_nan(absmax_nan(mxa, o0.x), o0.y), o1.x), o1.y);
                mxd = absmax_nan(absmax_nan(absmax_nan(absmax_nan(mxd, o0.x - c.x), o0.y - c.y), o1.x - c.z),
                                 o1.y - c.w);
            }
            if (ok[i][r]) *(float4 *)(out + o) = make_float4(o0.x, o0.y, o1.x, o1.y);
            if (MODE == kModeStepStore && ok[i][r]) {
                // checkpoint of the input pair (c = u^n, prev = u^{n-1}) in the encode kernel's
                // format: FP32 pair, or 16-bit a = c s_a and d = (c - prev) s_d
                const int64_t ci = (int64_t)shot * p.st_cstride + off + o;
                if (p.st_dtype == 0) {
                    *(float4 *)((float *)p.st_code + ci) = c;
                    if (p.st_comps == 2) *(float4 *)((float *)p.st_code + ci + p.field) = A;
                } else {
                    unsigned short *cc = (unsigned short *)p.st_code + ci;
                    *(uint2 *)cc = pack_code4(c, p.st_dtype, sca);
                    if (p.st_comps == 2)
                        *(uint2 *)(cc + p.field) =
                            pack_code4(make_float4(dc0.x, dc0.y, dc1.x, dc1.y), p.st_dtype, scd);
                }
            }
            if (MODE == kModeAdj && ok[i][r]) {
                // g += u^m * (L mu^{m+1});  at the source point g -= dt^2 w[m] mu^{m+1} / W
                const uint4 h = ur[i][r];
                const float4 u = afmt == 0 ? make_float4(__uint_as_float(h.x), __uint_as_float(h.y),
                                                         __uint_as_float(h.z), __uint_as_float(h.w))
                                           : unpack_code4(make_uint2(h.x, h.y), afmt, ainv);
                float2 g0 = __ffma2_rn(lo2(u), l0, lo2(gv[i][r]));
                float2 g1 = __ffma2_rn(hi2(u), l1, hi2(gv[i][r]));
                if (at_src) src_image(g0, g1, c, B, src_e, srcv);
                *(float4 *)(p.g + sb + o) = make_float4(g0.x, g0.y, g1.x, g1.y);
            }
        }
    if (MODE != kModeAdj && p.maxbits) {
        // the checkpoint codec's max-abs of the new state pair (u^{n+1}, u^n)
        const unsigned a = __reduce_max_sync(0xffffffffu, __float_as_uint(mxa) & 0x7fffffffu);
        const unsigned d = __reduce_max_sync(0xffffffffu, __float_as_uint(mxd) & 0x7fffffffu);
        if ((tid & 31) == 0) {
            if (a) atomicMax(p.maxbits + 2 * shot, a);
            if (d) atomicMax(p.maxbits + 2 * shot + 1, d);
        }
    }
}

template <int M, int MODE, bool ISO>
cudaError_t go(const Step3dParams &p, int nshots, const CUtensorMap &mid, const CUtensorMap &arm, cudaStream_t s)
{
    using C = Brick<M, MODE, ISO>;
    auto fn = MODE != kModeAdj && p.src_pts ? k_step3d_brick<M, MODE, ISO, MODE != kModeAdj>
                                            : k_step3d_brick<M, MODE, ISO, false>;
    cudaError_t e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    const int tz = (p.nz + C::TZ - 1) / C::TZ;
    const dim3 grid((p.nx + C::TX - 1) / C::TX, (p.ny + C::TY - 1) / C::TY, tz * nshots);
    return launch_pdl(fn, grid, dim3(C::NT), C::SMEM, s, p, mid, arm, tz);
}

template <int M, bool ISO>
cudaError_t go(const Step3dParams &p, int mode, int nshots, const CUtensorMap &mid, const CUtensorMap &arm,
               cudaStream_t s)
{
    if (mode == kModeStep) return go<M, kModeStep, ISO>(p, nshots, mid, arm, s);
    if (mode == kModeStepStore) return go<M, kModeStepStore, ISO>(p, nshots, mid, arm, s);
    return go<M, kModeAdj, ISO>(p, nshots, mid, arm, s);
}

}  // namespace

void brick_boxes(int M, int (&mid)[3], int (&arm)[3])
{
    using C = Brick<4, kModeStep, true>;   // the brick's extents are the same at both radii
    mid[0] = C::TX + 2 * M, mid[1] = C::TY + 2 * M, mid[2] = C::TZ;
    arm[0] = C::TX, arm[1] = C::TY, arm[2] = M;
}

// Bricks lie on a grid of x, y and z times shots, whose last two extents end at 65535.  Thin grids of
// many planes, rows or shots that exceed them stream (a one-dimensional grid).
static bool brick_grid_fits(const Step3dParams &p)
{
    using C = Brick<4, kModeStep, true>;   // the brick's extents are the same in every form
    const int64_t ty = (p.ny + C::TY - 1) / C::TY, tz = (p.nz + C::TZ - 1) / C::TZ;
    return ty <= 65535 && tz * p.nshots <= 65535;
}

// Whether a launch takes bricks: up to the points of all shots below which they measured
// faster than streaming (us, bricks / streaming).  Radius 4: forward 20.9 / 22.8 at 176^3
// computed points and 24.9 / 24.9 at 184^3, store 24.4 / 25.3 at 168^3 and 26.9 / 26.1 at 176^3,
// reverse 20.2 / 22.4 at 136^3, 22.2 / 22.3 at 144^3 and 24.9 / 24.5 at 152^3.  Radius 8: forward
// 34.1 / 34.8 at 192^3 and 47.6 / 47.3 at 208^3, store 30.7 / 32.9 at 168^3 and 34.5 / 33.7 at
// 176^3, reverse 27.4 / 32.3 at 160^3 and 40.2 / 36.7 at 168^3.  FWI_STEP3D_BRICK=0/1 overrides (1
// where the grid fits);
// the switches that choose among the streaming kernels turn bricks off.
bool step3d_use_brick(const Step3dParams &p, int mode)
{
    if (!brick_grid_fits(p)) return false;
    if (const char *e = std::getenv("FWI_STEP3D_BRICK")) return std::atoi(e) != 0;
    for (const char *v : {"FWI_STEP3D_TMEM", "FWI_STEP3D_VARIANT", "FWI_STEP3D_HALF", "FWI_STEP3D_TILE_G"})
        if (std::getenv(v)) return false;
    const double points = (double)p.nx * p.ny * p.nz * p.nshots;
    if (p.M == 4) return points <= (mode == kModeStep ? 6.0e6 : mode == kModeStepStore ? 5.0e6 : 3.0e6);
    return points <= (mode == kModeStep ? 8.5e6 : mode == kModeStepStore ? 5.2e6 : 4.3e6);
}

cudaError_t launch_step3d_brick(const Step3dParams &p, int mode, const CUtensorMap &mid,
                                const CUtensorMap &arm, cudaStream_t s)
{
    if (p.M == 8)
        return p.iso ? go<8, true>(p, mode, p.nshots, mid, arm, s) : go<8, false>(p, mode, p.nshots, mid, arm, s);
    if (p.M == 4)
        return p.iso ? go<4, true>(p, mode, p.nshots, mid, arm, s) : go<4, false>(p, mode, p.nshots, mid, arm, s);
    return cudaErrorInvalidValue;
}

}  // namespace fwi
