// 2-D time step on GB300 (sm_103a): halo tiles in shared memory, blocks of rows in registers.
//
// A CTA of two warps owns a tile of 128 columns by 2 RZ rows of one shot.  One thread asks
// the TMA unit for the tile with its halo of M columns and rows on every side (one 3-D box
// [shot][z][x]; zero fill outside the grid is the Dirichlet condition).  Meanwhile every
// thread loads the pointwise operands of its 4 columns x RZ rows (prev and W; the reverse
// step adds u^m, as FP32 or in place as a 16-bit checkpoint code, and g) straight into
// registers, so all of the CTA's bytes are in flight at once.  A thread then reads the
// RZ + 2M rows of its columns once, reads the side groups of each output row for the x-sums,
// and updates.  No queue moves from row to row, no thread waits for another after the tile
// has landed, and a small grid is spread over as many CTAs as it has tiles.
//
// DRAM bytes per point and step: 12 + 4 / shots forward (W is one field for all shots), 14 +
// 4 / shots with a 16-bit checkpoint store, 22 + 4 / shots reverse.  Measured on GB300
// against the kernel this replaces, which streamed rows through a register queue (86 to 98
// instructions a point, issue-bound; same results bit for bit), in us per step, forward /
// forward + store / reverse:
//   64 shots of 440 x 1064, radius 4:  95.1 / 115.3 / 120.0  ->  67.5 / 79.3 / 108.1
//   the same at radius 8:             146.1 / 158.3 / 169.7  ->  73.5 / 85.2 / 114.2
//   one shot of 557 x 940, radius 8:   21.2 /  23.2 /  37.1  ->   7.9 /  8.4 /   8.1
//   one shot of 241 x 241, radius 4:   12.7 /  14.9 /  20.6  ->   6.2 /  6.3 /   8.0
// (5.4 / 5.3 / 6.1 TB/s on the first line; the last two hold a few us of event overhead).
// What bounds it: the latency of a CTA's loads.  Its load phase and its arithmetic do not
// overlap, what hides one is the SM's other CTAs, and registers cap those: 14.4 warps an SM,
// issue slots 48 % and the L1 data pipe 49 % busy.  It is not DRAM: 16 shots, whose fields stay
// in L2, take the same time per point (18.5 us).  A persistent pipeline of 128 x 32 tiles, all
// operands by TMA in a ring of two stages, two CTAs of 8 warps an SM, gave the forward step 70.3
// -> 66.4 us but the storing one 84.2 -> 84.4, radius 8 76.0 -> 87.6 and 16 shots 18.5 -> 21.1;
// rows of a later tile prefetched into L2 gave 2 % forward and took 2 % in reverse.
//
// Tile: two warps of 4 rows, eight CTAs per SM (forward modes), or of 3 rows (reverse, which
// holds twice the operands).  Measured at radius 4, forward / store / reverse: 2 warps x 2
// rows 75.3 / 81.2 / 119.7, 1 x 4 67.6 / 79.3 / 109.4, 2 x 3 76.2 / 89.2 / 108.1, 2 x 4 67.5 /
// 79.3 / 118.5; at radius 8 2 x 4 73.5 / 85.2 / 134.2, 1 x 4 85.1 / 99.5 / 117.3, 2 x 3 83.0 /
// 95.0 / 114.2.  Larger CTAs (4 x 2, 8 x 2, 8 x 4) were slower than 2 x 2 in an earlier form.
#include <cuda.h>

#include <algorithm>

#include "code16.cuh"
#include "fwi_internal.h"
#include "k_step3d.cuh"
#include "pdl.cuh"
#include "step2d_math.cuh"
#include "taps.cuh"

namespace fwi {
namespace {

using s2d::hi2;
using s2d::lap_x;
using s2d::lo2;
using s2d::update4;
using s2d::z_block;
using s3d::absmax_nan;
using s3d::mbar_expect_tx;
using s3d::mbar_init;
using s3d::mbar_wait;
using s3d::smem_u32;

constexpr int kTileX = 128;   // columns per tile: one warp, four points per lane
enum { kStep = 0, kStore = 1, kImg = 2 };

__device__ __forceinline__ void tma_tile(void *dst, const CUtensorMap *map, int x, int z, int shot,
                                         uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(z), "r"(shot), "r"(smem_u32(bar))
        : "memory");
}

// Warps and CTAs per SM, and rows per thread of each mode (see above); tile rows a launch holds.
constexpr int kWarps = 2, kMinCtas = 8;
constexpr int kGridYMax = 65535;
__host__ __device__ constexpr int tile_rz(int mode) { return mode == kImg ? 3 : 4; }

// TAPS: an off-grid source is added too.  MORE: the launch starts at tile row row0 (else 0).  Both
// are instantiations of their own, so that the common one pays nothing for them (3 % and 0.5 % of a
// 64-shot step).
template <int M, int MODE, bool TAPS, bool MORE>
__global__ void __launch_bounds__(32 * kWarps, kMinCtas)
k_step2d_tile(const __grid_constant__ StepParams p, const __grid_constant__ CUtensorMap map, int row0)
{
    constexpr int RZ = tile_rz(MODE), TZ = kWarps * RZ, SX = kTileX + 2 * M, SZ = TZ + 2 * M;
    __shared__ __align__(128) float tile[SZ][SX];
    __shared__ __align__(8) uint64_t bar;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int shot = blockIdx.z, nz = p.g.nz, nx = p.g.nx;
    pdl_next();
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    const int tz = (MORE ? row0 : 0) + blockIdx.y;             // tile row
    const int x0 = blockIdx.x * kTileX + 4 * lane, zr = tz * TZ + warp * RZ;
    const bool xin = x0 < nx;
    const int plane = (int)p.g.plane;
    const int64_t off = (int64_t)zr * plane + x0;              // row zr, column x0
    const int64_t sb = (int64_t)shot * p.g.field + off;
    float *prev = p.prev + sb;
    const float *__restrict__ Wp = p.W + off;
    const int afmt = p.aux_fmt;
    const int left = xin ? nz - zr : 0;                        // rows of this block in the grid
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 pv[RZ], Wv[RZ], gv[MODE == kImg ? RZ : 1];
    uint4 ur[MODE == kImg ? RZ : 1];
    float *gp = MODE == kImg ? p.gacc + sb : nullptr;
    const char *up =
        MODE == kImg ? (const char *)p.aux + ((int64_t)shot * p.aux_stride + off) * (afmt ? 2 : 4) : nullptr;
    float sz[RZ];
#pragma unroll
    for (int r = 0; r < RZ; ++r) {
        Wv[r] = r < left ? __ldg((const float4 *)(Wp + r * plane)) : zero4;
        sz[r] = __ldg(p.sig_z + min(zr + r, nz - 1));
    }
    const float4 sx4 = xin ? __ldg((const float4 *)(p.sig_x + x0)) : zero4;   // padded with zeros
    pdl_wait();
    if (threadIdx.x == 0) {
        mbar_expect_tx(&bar, SX * SZ * 4);
        tma_tile(&tile[0][0], &map, blockIdx.x * kTileX - M, tz * TZ - M, shot, &bar);
    }
#pragma unroll
    for (int r = 0; r < RZ; ++r) {
        pv[r] = r < left ? *(const float4 *)(prev + r * plane) : zero4;
        if (MODE == kImg) {
            gv[r] = r < left ? *(const float4 *)(gp + r * plane) : zero4;
            ur[r] = make_uint4(0u, 0u, 0u, 0u);
            if (r < left) {
                if (afmt == 0) {
                    ur[r] = *(const uint4 *)(up + (int64_t)r * plane * 4);
                } else {
                    const uint2 h = *(const uint2 *)(up + (int64_t)r * plane * 2);
                    ur[r].x = h.x;
                    ur[r].y = h.y;
                }
            }
        }
    }
    const int n = (p.n_dev ? *p.n_dev : 0) + p.n;
    int src_r = -1, src_e = 0;
    float srcv = 0.0f;
    if (p.src_off) {
        // the source in this thread's block?  (one test per warp for almost all of them)
        const int64_t d = p.src_off[shot] - (off - 4 * lane);
        if (d >= 0 && d < (int64_t)RZ * plane) {
            const int r = (int)(d / plane), e = (int)d - r * plane - 4 * lane;
            if (e >= 0 && e < 4 && xin) {
                src_r = r;
                src_e = e;
                srcv = p.dt2 * p.wavelet[(int64_t)shot * p.nt + n];
            }
        }
    }
    bool taps = false;   // an off-grid source's taps meet this thread's block
    if (TAPS && left > 0) {
        taps = taps_meet(p.src_pts[shot], 2, zr, RZ, 0, 1, x0);
        if (taps) srcv = p.dt2 * p.wavelet[(int64_t)shot * p.nt + n];
    }
    float sca = 1.0f, scd = 1.0f;
    char *codes = nullptr;
    if (MODE == kStore) {
        codes = (char *)p.st_code + ((int64_t)shot * p.st_cstride + off) * (p.st_dtype ? 2 : 4);
        if (p.st_dtype != 0) {
            const float2 sc = store_scales(p.st_max, shot, p.st_dtype);
            sca = sc.x;
            scd = sc.y;
        }
    }
    const float ainv = (MODE == kImg && p.aux_scale) ? 1.0f / p.aux_scale[2 * shot] : 1.0f;
    if (MODE != kImg && threadIdx.x == 0 && blockIdx.x == 0 && tz == 0)
        store_bookkeeping(p.st_max, shot, p.st_dtype, p.st_scale, p.err, p.max_clear);
    __syncthreads();   // the barrier is initialised
    const bool ok = mbar_wait(&bar, 0);
    if (!ok) {
        // a bounded wait gave up: report, then give the copy a bounded chance to land
        // before the CTA's shared memory is released
        if (threadIdx.x == 0) atomicOr(p.err, 2u);
        (void)mbar_wait(&bar, 0);
        return;
    }

    float2 za[RZ], zb[RZ];
    float4 ctr[RZ];
    const float *col = &tile[warp * RZ][M + 4 * lane];
    z_block<M, RZ>(col, SX, p.c, ctr, za, zb);
    float mxa = 0.0f, mxd = 0.0f;
#pragma unroll
    for (int r = 0; r < RZ; ++r) {
        const bool in = r < left;
        float w[4 + 2 * M];
        const float *row = col + (r + M) * SX - M;
#pragma unroll
        for (int g4 = 0; g4 < (4 + 2 * M) / 4; ++g4) {
            const float4 v = g4 == M / 4 ? ctr[r] : *(const float4 *)(row + 4 * g4);
            w[4 * g4] = v.x, w[4 * g4 + 1] = v.y, w[4 * g4 + 2] = v.z, w[4 * g4 + 3] = v.w;
        }
        float2 l0, l1;
        lap_x<M>(w, ctr[r], p.c, za[r], zb[r], l0, l1);
        const float4 c = ctr[r];
        float4 o = update4(c, l0, l1, pv[r], Wv[r], sx4, sz[r], (MODE != kImg && r == src_r) ? src_e : -1, srcv);
        if (TAPS && taps && in) add_taps(p.src_pts[shot], 2, zr + r, 0, x0, srcv, sz[r], sx4, o);
        if (p.rec_map && zr + r == p.rec_z && xin) {
            const int4 ri = __ldg((const int4 *)(p.rec_map + (int64_t)shot * plane + x0));
            const int idx[4] = {ri.x, ri.y, ri.z, ri.w};
            float ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (idx[e] < 0) continue;
                if (MODE != kImg)
                    p.rec_tr[((int64_t)shot * p.nt + n) * p.nrec + idx[e]] = ov[e];
                else
                    ov[e] = __fadd_rn(ov[e], __fmul_rn(p.inj_scale[(int64_t)shot * p.nrec + idx[e]],
                                                       p.inj_q[((int64_t)shot * p.nt + p.inj_n) * p.nrec + idx[e]]));
            }
            if (MODE == kImg) o = make_float4(ov[0], ov[1], ov[2], ov[3]);
        }
        if (in) *(float4 *)(prev + r * plane) = o;
        if (MODE == kStore && in) {
            // FP32 pair unchanged, or 16-bit a = c s_a and d = (c - prev) s_d
            if (p.st_dtype == 0) {
                float *cc = (float *)codes + r * plane;
                *(float4 *)cc = c;
                if (p.st_comps == 2) *(float4 *)(cc + p.g.field) = pv[r];
            } else {
                unsigned short *cc = (unsigned short *)codes + r * plane;
                *(uint2 *)cc = pack_code4(c, p.st_dtype, sca);
                if (p.st_comps == 2)
                    *(uint2 *)(cc + p.g.field) = pack_code4(
                        make_float4(c.x - pv[r].x, c.y - pv[r].y, c.z - pv[r].z, c.w - pv[r].w),
                        p.st_dtype, scd);
            }
        }
        if (MODE != kImg && p.maxbits) {
            mxa = absmax_nan(absmax_nan(absmax_nan(absmax_nan(mxa, o.x), o.y), o.z), o.w);
            mxd = absmax_nan(absmax_nan(absmax_nan(absmax_nan(mxd, o.x - c.x), o.y - c.y), o.z - c.z),
                             o.w - c.w);
        }
        if (MODE == kImg && in) {
            // g += u^m (L mu^{m+1});  at the source point g -= dt^2 w[m] mu^{m+1} / W
            const float4 u = afmt == 0 ? make_float4(__uint_as_float(ur[r].x), __uint_as_float(ur[r].y),
                                                     __uint_as_float(ur[r].z), __uint_as_float(ur[r].w))
                                       : unpack_code4(make_uint2(ur[r].x, ur[r].y), afmt, ainv);
            float2 g0 = __ffma2_rn(lo2(u), l0, lo2(gv[r]));
            float2 g1 = __ffma2_rn(hi2(u), l1, hi2(gv[r]));
            if (r == src_r) s3d::src_image(g0, g1, c, Wv[r], src_e, srcv);
            *(float4 *)(gp + r * plane) = make_float4(g0.x, g0.y, g1.x, g1.y);
        }
    }
    if (MODE != kImg && p.maxbits) {
        // the checkpoint codec's max-abs of the new state pair (u^{n+1}, u^n)
        const unsigned a = __reduce_max_sync(0xffffffffu, __float_as_uint(mxa) & 0x7fffffffu);
        const unsigned d = __reduce_max_sync(0xffffffffu, __float_as_uint(mxd) & 0x7fffffffu);
        if (lane == 0) {
            if (a) atomicMax(p.maxbits + 2 * shot, a);
            if (d) atomicMax(p.maxbits + 2 * shot + 1, d);
        }
    }
}

template <int M, int MODE>
cudaError_t go(const StepParams &p, int nshots, const CUtensorMap &map, cudaStream_t s)
{
    constexpr int TZ = kWarps * tile_rz(MODE);
    auto *first = MODE != kImg && p.src_pts ? k_step2d_tile<M, MODE, MODE != kImg, false>
                                            : k_step2d_tile<M, MODE, false, false>;
    auto *more = MODE != kImg && p.src_pts ? k_step2d_tile<M, MODE, MODE != kImg, true>
                                           : k_step2d_tile<M, MODE, false, true>;
    // tile rows on grid.y, at most 65535 a launch (a launch writes its own rows of prev only)
    const int rows = (p.g.nz + TZ - 1) / TZ;
    cudaError_t e = cudaSuccess;
    for (int row0 = 0; row0 < rows && e == cudaSuccess; row0 += kGridYMax) {
        const dim3 grid((p.g.nx + kTileX - 1) / kTileX, std::min(rows - row0, kGridYMax), nshots);
        e = launch_pdl(row0 ? more : first, grid, dim3(32 * kWarps), 0, s, p, map, row0);
    }
    return e;
}

}  // namespace

int step2d_tile_cols() { return kTileX; }

int step2d_tile_rows(bool img) { return kWarps * tile_rz(img ? kImg : kStep); }

cudaError_t launch_step2d_tile(const StepParams &p, int nshots, bool img, const CUtensorMap &map,
                               cudaStream_t s)
{
    if (p.g.M == 4)
        return img ? go<4, kImg>(p, nshots, map, s)
                   : p.st_code ? go<4, kStore>(p, nshots, map, s) : go<4, kStep>(p, nshots, map, s);
    if (p.g.M == 8)
        return img ? go<8, kImg>(p, nshots, map, s)
                   : p.st_code ? go<8, kStore>(p, nshots, map, s) : go<8, kStep>(p, nshots, map, s);
    return cudaErrorInvalidValue;
}

}  // namespace fwi
