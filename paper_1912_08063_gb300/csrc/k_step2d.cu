// The 2-D forward kernels of the serving loop's shared launch: the multi-request step
// (register z-streaming with L1-served x-windows) and the on-chip temporal blocking of
// small grids.  Their arithmetic is that of every 2-D step (step2d_math.cuh).
//
// Multi-request step: a CTA streams along z over rows of a 256-wide x tile (64 threads x 4
// points).  Each thread keeps the 2M + 1 rows of its four points in a register queue
// (z-neighbours) and reads the x-window of the output row (M floats either side, in 16-byte
// groups) straight from global memory: the row was read by the neighbouring threads a few
// iterations earlier, so those loads hit L1/L2, and the kernel needs neither shared memory
// nor barriers.
#include <cooperative_groups.h>

#include "fwi_internal.h"
#include "step2d_math.cuh"

namespace fwi {

namespace {

constexpr int kThreads2 = 64;            // threads per CTA
constexpr int kTile2 = 4 * kThreads2;    // x points per CTA

__device__ __forceinline__ float4 ld4(const float *__restrict__ f, int64_t row, int x,
                                      int px, bool zin)
{
    // x is a multiple of 4; groups outside [0, px) and rows outside the grid read as zero
    if (!zin || x < 0 || x >= px) return make_float4(0.f, 0.f, 0.f, 0.f);
    return __ldg((const float4 *)(f + row + x));
}

using namespace s2d;

// Global operands of one output row: the row entering the z-queue, the x-window groups
// left and right of the centre, and the pointwise values.
template <int M>
struct RowIn {
    float4 qn, win[2 * (M / 4)], pv, Wv;
};

// One CTA's work: x tile bx, z-chunk zc of the request p, from state (cur = u^n,
// prev = u^{n-1}, overwritten by u^{n+1}) at step n.  The global loads of row z + 1 are
// issued before row z's arithmetic.  With row_tr, the receivers are the rn consecutive
// nodes of row rz from column rx0 on, and the epilogue writes their samples u^{n+1} to
// row_tr[0 .. rn).
template <int M>
__device__ __forceinline__ void step2d_body(const StepParams &p, const float *__restrict__ cur,
                                            float *__restrict__ prev, int n, int bx, int zc,
                                            float *row_tr, int rz, int rx0, int rn)
{
    constexpr int Q = 2 * M + 1, W4 = M / 4;   // x-window: W4 groups of 4 either side
    const int nz = p.g.nz, nx = p.g.nx, px = p.g.px;
    const int z0 = zc * p.zchunk, z1 = min(nz, z0 + p.zchunk);
    const int x0 = bx * kTile2 + threadIdx.x * 4;
    const bool xin = x0 < nx;
    const int64_t plane = p.g.plane;

    float4 q[Q];
#pragma unroll
    for (int i = 0; i < Q - 1; ++i) {
        const int z = z0 - M + i;
        const bool zin = z >= 0 && z < nz;
        q[i] = ld4(cur, (int64_t)z * plane, x0, px, zin);
    }
    const float4 sx = xin ? __ldg((const float4 *)(p.sig_x + x0)) : make_float4(0.f, 0.f, 0.f, 0.f);
    int src_z = -1, src_e = 0;
    float srcv = 0.0f;
    if (p.src_off) {
        const int64_t s = p.src_off[0];
        const int sz = (int)(s / plane), sxx = (int)(s - (int64_t)sz * plane);
        if (sxx >= x0 && sxx < x0 + 4) {
            src_z = sz;
            src_e = sxx - x0;
            srcv = p.dt2 * p.wavelet[n];
        }
    }

    auto load_row = [&](int z, RowIn<M> &in) {
        const int zn = z + M;
        const int64_t row = (int64_t)z * plane;
        in.qn = ld4(cur, (int64_t)zn * plane, x0, px, zn < nz);
#pragma unroll
        for (int j = 0; j < 2 * W4; ++j) {
            const int g4 = j < W4 ? j : j + 1;
            in.win[j] = ld4(cur, row, x0 + 4 * (g4 - W4), px, true);
        }
        if (xin) {
            in.pv = __ldg((const float4 *)(prev + row + x0));
            in.Wv = __ldg((const float4 *)(p.W + row + x0));
        }
    };
    RowIn<M> nxt;
    if (z0 < z1) load_row(z0, nxt);
    for (int z = z0; z < z1; ++z) {
        const RowIn<M> in = nxt;
        if (z + 1 < z1) load_row(z + 1, nxt);
        q[Q - 1] = in.qn;
        const int64_t row = (int64_t)z * plane;
        // x-window of the output row: groups x0 - M .. x0 + 3 + M
        float w[4 + 2 * M];
#pragma unroll
        for (int g4 = 0; g4 < 2 * W4 + 1; ++g4) {
            const float4 v = (g4 == W4) ? q[M] : in.win[g4 < W4 ? g4 : g4 - 1];
            w[4 * g4] = v.x, w[4 * g4 + 1] = v.y, w[4 * g4 + 2] = v.z, w[4 * g4 + 3] = v.w;
        }
        float2 l0, l1;
        lap4<M>(w, q, p.c, l0, l1);
        if (xin) {
            const float4 o = update4(q[M], l0, l1, in.pv, in.Wv, sx, p.sig_z[z],
                                     z == src_z ? src_e : -1, srcv);
            *(float4 *)(prev + row + x0) = o;
            if (row_tr && z == rz) {
                const float rhs[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = x0 + e - rx0;
                    if (r >= 0 && r < rn) row_tr[r] = rhs[e];
                }
            }
        }
#pragma unroll
        for (int i = 0; i < Q - 1; ++i) q[i] = q[i + 1];
    }
}

// ---- the serving loop's shared launch: one forward step of every request in a table ----

// Step t of a tick for every request of the table: work item w of the persistent loop is
// (x tile, z-chunk) (w - work0) of the entry whose range holds it; the entry's state is
// (u0, u1) at the tick's start, so step t reads u^n from u0 (t even) or u1 (t odd) and
// overwrites the other; entries whose nt ends within the tick skip the steps past it.
template <int M>
__global__ void __launch_bounds__(kThreads2) k_step2d_multi(const Batch2d *__restrict__ tab, int t)
{
    const int count = tab->count, total = tab->total_work;
    int e = 0;
    for (int w = blockIdx.x; w < total; w += gridDim.x) {
        while (e + 1 < count && tab->e[e + 1].work0 <= w) ++e;   // w increases: scan on
        const Batch2dEntry &E = tab->e[e];
        const int n = E.n0 + t;
        if (n >= E.p.nt) continue;
        const int lw = w - E.work0;
        const int bx = lw % E.xtiles, zc = lw / E.xtiles;
        const bool odd = t & 1;
        step2d_body<M>(E.p, odd ? E.u1 : E.u0, odd ? E.u0 : E.u1, n, bx, zc,
                       E.rec_z >= 0 ? E.traces + (int64_t)n * E.nrec : nullptr, E.rec_z, E.rec_x0,
                       E.nrec);
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

// ---- temporal blocking on chip: one thread-block cluster per request ----
//
// A small 2-D request is advanced by k steps in one launch.  Its C CTAs (one cluster)
// split the nz rows into bands [r0, r1); each CTA holds its band of u^n and u^{n-1} in
// shared memory for the whole launch, reads the M halo rows above and below from its
// neighbours' shared memory (distributed shared memory of the cluster), and writes
// u^{n+1} over its u^{n-1} band; a cluster barrier separates the steps (hardware, no
// polling).  W, the sponge tables and the wavelet are read from global memory (L2).
// Receivers that form one row are sampled in the epilogue; the source is added by the
// thread owning its node.  The arithmetic of a point is the single step's (lap4,
// update4 on the same operands), so k steps here equal k single steps bit for bit.  The
// states return to global memory at the end of the launch (buffer 0 to u0, 1 to u1, the
// same parity the single steps leave).
constexpr int kClThreads = 512;

template <int M>
__global__ void __launch_bounds__(kClThreads, 1) k_step2d_cluster(const Batch2d *__restrict__ tab, int k)
{
    namespace cg = cooperative_groups;
    constexpr int Q = 2 * M + 1, W4 = M / 4;
    extern __shared__ __align__(16) float smc[];
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int req = blockIdx.x / C;   // one cluster per request (uniform per cluster)
    if (req >= tab->count) return;
    const Batch2dEntry &E = tab->e[req];
    const StepParams &p = E.p;
    const int nz = p.g.nz, nx = p.g.nx, px = p.g.px;
    const int r0 = (int)((int64_t)rank * nz / C), r1 = (int)((int64_t)(rank + 1) * nz / C);
    const int rup = rank > 0 ? (int)((int64_t)(rank - 1) * nz / C) : 0;   // first row above
    const int R = r1 - r0, band = (nz + C - 1) / C * px;   // floats per band buffer
    float *b0 = smc, *b1 = smc + band;
    const int G = px / 4;
    for (int i = threadIdx.x; i < R * G; i += blockDim.x) {
        *(float4 *)(b0 + 4 * i) = __ldg((const float4 *)(E.u0 + (int64_t)r0 * px) + i);
        *(float4 *)(b1 + 4 * i) = __ldg((const float4 *)(E.u1 + (int64_t)r0 * px) + i);
    }
    // source node
    int src_z = -1, src_x = -1;
    if (p.src_off) {
        const int64_t so = p.src_off[0];
        src_z = (int)(so / px);
        src_x = (int)(so - (int64_t)src_z * px);
    }
    cl.sync();
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 0; s < k; ++s) {
        const int n = E.n0 + s;
        if (n >= p.nt) break;   // the same for every CTA of the cluster
        const float *cur = (s & 1) ? b1 : b0;
        float *prv = (s & 1) ? b0 : b1;
        const float *up = rank > 0 ? cl.map_shared_rank(cur, rank - 1) : nullptr;
        const float *dn = rank < C - 1 ? cl.map_shared_rank(cur, rank + 1) : nullptr;
        const float srcv = p.dt2 * p.wavelet[n];
        float *row_tr = E.rec_z >= r0 && E.rec_z < r1 ? E.traces + (int64_t)n * E.nrec : nullptr;
        for (int it = threadIdx.x; it < R * G; it += blockDim.x) {
            const int lr = it / G, g = it - lr * G;
            const int z = r0 + lr, x0 = 4 * g;
            if (x0 >= nx) continue;
            float4 q[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const int zz = z - M + i;
                const float *src = zz < 0 || zz >= nz ? nullptr
                                   : zz < r0          ? up + (int64_t)(zz - rup) * px
                                   : zz >= r1         ? dn + (int64_t)(zz - r1) * px
                                                      : cur + (int64_t)(zz - r0) * px;
                q[i] = src ? *(const float4 *)(src + x0) : zero4;
            }
            float w[4 + 2 * M];
            const float *rowc = cur + (int64_t)lr * px;
#pragma unroll
            for (int g4 = 0; g4 < 2 * W4 + 1; ++g4) {
                const int xg = x0 + 4 * (g4 - W4);
                const float4 v = g4 == W4 ? q[M] : (xg < 0 || xg >= px ? zero4 : *(const float4 *)(rowc + xg));
                w[4 * g4] = v.x, w[4 * g4 + 1] = v.y, w[4 * g4 + 2] = v.z, w[4 * g4 + 3] = v.w;
            }
            float2 l0, l1;
            lap4<M>(w, q, p.c, l0, l1);
            const float4 sx = __ldg((const float4 *)(p.sig_x + x0));
            const float4 pv = *(const float4 *)(prv + (int64_t)lr * px + x0);
            const float4 Wv = __ldg((const float4 *)(p.W + (int64_t)z * px + x0));
            const int se = (z == src_z && src_x >= x0 && src_x < x0 + 4) ? src_x - x0 : -1;
            const float4 o = update4(q[M], l0, l1, pv, Wv, sx, p.sig_z[z], se, srcv);
            *(float4 *)(prv + (int64_t)lr * px + x0) = o;
            if (row_tr && z == E.rec_z) {
                const float rhs[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int r = x0 + e - E.rec_x0;
                    if (r >= 0 && r < E.nrec) row_tr[r] = rhs[e];
                }
            }
        }
        // every band's u^{n+1} is written and every read of u^n is done
        cl.sync();
    }
    for (int i = threadIdx.x; i < R * G; i += blockDim.x) {
        ((float4 *)(E.u0 + (int64_t)r0 * px))[i] = *(const float4 *)(b0 + 4 * i);
        ((float4 *)(E.u1 + (int64_t)r0 * px))[i] = *(const float4 *)(b1 + 4 * i);
    }
}

int cluster2d_max_smem() { return 220 * 1024; }

int cluster2d_size(int M)
{
    // the largest cluster (16, else 8) of which at least one fits with full shared memory
    const void *fn = M == 8 ? (const void *)k_step2d_cluster<8> : (const void *)k_step2d_cluster<4>;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, cluster2d_max_smem()) !=
            cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    for (int C : {16, 8}) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(C, 1, 1);
        cfg.blockDim = dim3(kClThreads, 1, 1);
        cfg.dynamicSmemBytes = cluster2d_max_smem();
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, fn, &cfg) == cudaSuccess && nc > 0) return C;
        cudaGetLastError();
    }
    return 0;
}

cudaError_t launch_step2d_cluster(const Batch2d *tab, int M, int k, int C, int nreq, int smem,
                                  cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(C * (nreq > 0 ? nreq : 1), 1, 1);
    cfg.blockDim = dim3(kClThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (M == 4) return cudaLaunchKernelEx(&cfg, k_step2d_cluster<4>, tab, k);
    if (M == 8) return cudaLaunchKernelEx(&cfg, k_step2d_cluster<8>, tab, k);
    return cudaErrorInvalidValue;
}

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
