// The multi-request 2-D forward step of the serving loop's shared launch: the halo tiles of the
// single step (k_step2d_tile.cu) for every request of a table, with its arithmetic
// (step2d_math.cuh), so results are the same bit for bit.  The table's fields have no tensor maps;
// a tile and its halo come by 16-byte asynchronous copies, zeros outside the grid.  Bound by the
// latency of a tile's loads, like the single step.  Measured on GB300 against the kernel it
// replaces, which streamed rows of 256 columns through a register queue, ms for a stream of
// forward requests of 600 steps: one of 560^2 5.3 -> 4.1 (radius 8 7.9 -> 4.2), four 8.8 -> 7.3
// (11.8 -> 7.0), twelve 17.1 -> 16.2 (21.4 -> 18.4), eight of 940^2 22.6 -> 21.1 (28.7 -> 26.1).
// Eight CTAs an SM at radius 4 and six at radius 8, where eight would spill; six at radius 4 took
// 17.9 for the twelve and 23.8 for the eight.
#include "fwi_internal.h"
#include "k_step3d.cuh"
#include "step2d_math.cuh"

namespace fwi {

namespace {

using s2d::lap_x;
using s2d::update4;
using s2d::z_block;
using s3d::smem_u32;

constexpr int kThreads2 = 64;            // threads per CTA: two warps
constexpr int kTile2 = 128;              // columns per tile: four points per lane
constexpr int kRows2 = 4;                // rows per thread
static_assert(2 * kRows2 == kMultiRows && kTile2 == kMultiCols, "work items");

// One tile of the request p: tile (bx, bz) from state (cur = u^n, prev = u^{n-1}, overwritten by
// u^{n+1}) at step n.  With row_tr, the receivers are the rn consecutive nodes of row rz from
// column rx0 on, and the epilogue writes their samples u^{n+1} to row_tr[0 .. rn).
template <int M>
__device__ __forceinline__ void step2d_tile(const StepParams &p, float *tile, const float *__restrict__ cur,
                                            float *__restrict__ prev, int n, int bx, int bz, float *row_tr, int rz,
                                            int rx0, int rn)
{
    constexpr int SX = kTile2 + 2 * M, SZ = 2 * kRows2 + 2 * M, GX = SX / 4;
    const int nz = p.g.nz, nx = p.g.nx, px = p.g.px, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t plane = p.g.plane;
    __syncthreads();   // both warps are done with the tile before
    for (int i = threadIdx.x; i < GX * SZ; i += kThreads2) {
        const int r = i / GX, g = i - r * GX, z = bz * 2 * kRows2 - M + r, x = bx * kTile2 - M + 4 * g;
        const bool in = z >= 0 && z < nz && x >= 0 && x < px;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(tile + r * SX + 4 * g)),
                     "l"(in ? cur + z * plane + x : cur), "r"(in ? 16 : 0)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int x0 = bx * kTile2 + 4 * lane, zr = bz * 2 * kRows2 + warp * kRows2;
    const int left = x0 < nx ? nz - zr : 0;   // rows of this thread's block in the grid
    const int64_t off = zr * plane + x0;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 pv[kRows2], Wv[kRows2];
    float sz[kRows2];
#pragma unroll
    for (int r = 0; r < kRows2; ++r) {
        pv[r] = r < left ? *(const float4 *)(prev + off + r * plane) : zero4;
        Wv[r] = r < left ? __ldg((const float4 *)(p.W + off + r * plane)) : zero4;
        sz[r] = __ldg(p.sig_z + min(zr + r, nz - 1));
    }
    const float4 sx = left > 0 ? __ldg((const float4 *)(p.sig_x + x0)) : zero4;
    int src_r = -1, src_e = 0;
    float srcv = 0.0f;
    if (p.src_off) {
        const int64_t s = p.src_off[0];
        const int r = (int)(s / plane) - zr, e = (int)(s % plane) - x0;
        if (r >= 0 && r < kRows2 && e >= 0 && e < 4) {
            src_r = r;
            src_e = e;
            srcv = p.dt2 * p.wavelet[n];
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const float *col = tile + warp * kRows2 * SX + M + 4 * lane;
    float2 za[kRows2], zb[kRows2];
    float4 ctr[kRows2];
    z_block<M, kRows2>(col, SX, p.c, ctr, za, zb);
#pragma unroll
    for (int r = 0; r < kRows2; ++r) {
        float w[4 + 2 * M];
        const float *row = col + (r + M) * SX - M;
#pragma unroll
        for (int g4 = 0; g4 < (4 + 2 * M) / 4; ++g4) {
            const float4 v = g4 == M / 4 ? ctr[r] : *(const float4 *)(row + 4 * g4);
            w[4 * g4] = v.x, w[4 * g4 + 1] = v.y, w[4 * g4 + 2] = v.z, w[4 * g4 + 3] = v.w;
        }
        float2 l0, l1;
        lap_x<M>(w, ctr[r], p.c, za[r], zb[r], l0, l1);
        const float4 o = update4(ctr[r], l0, l1, pv[r], Wv[r], sx, sz[r], r == src_r ? src_e : -1, srcv);
        if (r < left) {
            *(float4 *)(prev + off + r * plane) = o;
            if (row_tr && zr + r == rz) {
                const float v[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int k = x0 + e - rx0;
                    if (k >= 0 && k < rn) row_tr[k] = v[e];
                }
            }
        }
    }
}

// ---- the serving loop's shared launch: one forward step of every request in a table ----

// Step t of a tick for every request of the table: work item w of the persistent loop is
// (x tile, z tile) (w - work0) of the entry whose range holds it; the entry's state is
// (u0, u1) at the tick's start, so step t reads u^n from u0 (t even) or u1 (t odd) and
// overwrites the other; entries whose nt ends within the tick skip the steps past it.
template <int M>
__global__ void __launch_bounds__(kThreads2, M == 8 ? 6 : 8) k_step2d_multi(const Batch2d *__restrict__ tab, int t)
{
    __shared__ __align__(16) float tile[(2 * kRows2 + 2 * M) * (kTile2 + 2 * M)];
    const int count = tab->count, total = tab->total_work;
    int e = 0;
    for (int w = blockIdx.x; w < total; w += gridDim.x) {
        while (e + 1 < count && tab->e[e + 1].work0 <= w) ++e;   // w increases: scan on
        const Batch2dEntry &E = tab->e[e];
        const int n = E.n0 + t;
        if (n >= E.p.nt) continue;
        const int lw = w - E.work0;
        const int bx = lw % E.xtiles, bz = lw / E.xtiles;
        const bool odd = t & 1;
        step2d_tile<M>(E.p, tile, odd ? E.u1 : E.u0, odd ? E.u0 : E.u1, n, bx, bz,
                       E.rec_z >= 0 ? E.traces + (int64_t)n * E.nrec : nullptr, E.rec_z, E.rec_x0, E.nrec);
    }
}

// The receiver samples of step t, traces[n][r] = u^{n+1}(rec_r), of every entry whose
// step does not sample them itself (nsamp receivers each).
__global__ void k_sample_multi(const Batch2d *__restrict__ tab, int t)
{
    const int count = tab->count, total = tab->total_rec;
    int e = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        while (e + 1 < count && tab->e[e + 1].rec0 <= i) ++e;
        const Batch2dEntry &E = tab->e[e];
        const int n = E.n0 + t;
        if (n >= E.p.nt) continue;
        const int r = i - E.rec0;
        const float *next = (t & 1) ? E.u0 : E.u1;   // the buffer step t wrote
        E.traces[(int64_t)n * E.nrec + r] = next[E.rec_off[r]];
    }
}

}  // namespace

int multi2d_grid(int M)
{
    int dev = 0, sms = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per, M == 8 ? (const void *)k_step2d_multi<8> : (const void *)k_step2d_multi<4>,
            kThreads2, 0) != cudaSuccess) {
        cudaGetLastError();
        return 152 * 8;
    }
    return (sms > 0 ? sms : 152) * (per > 0 ? per : 1);
}

cudaError_t launch_step2d_multi(const Batch2d *tab, int M, int t, int grid, cudaStream_t s)
{
    if (M == 4) k_step2d_multi<4><<<grid, kThreads2, 0, s>>>(tab, t);
    else if (M == 8) k_step2d_multi<8><<<grid, kThreads2, 0, s>>>(tab, t);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_sample_multi(const Batch2d *tab, int t, int grid, cudaStream_t s)
{
    k_sample_multi<<<grid, 256, 0, s>>>(tab, t);
    return cudaGetLastError();
}

}  // namespace fwi
