// The multi-request 2-D forward step of the serving loop's shared launch, with the arithmetic
// of every 2-D step (step2d_math.cuh): a CTA streams along z over rows of a 256-wide x tile (64 threads x 4
// points).  Each thread keeps the 2M + 1 rows of its four points in a register queue
// (z-neighbours) and reads the x-window of the output row (M floats either side, in 16-byte
// groups) straight from global memory: the row was read by the neighbouring threads a few
// iterations earlier, so those loads hit L1/L2, and the kernel needs neither shared memory
// nor barriers.
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
