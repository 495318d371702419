// Off-grid sources and receivers: sampling, injection and the point terms of the
// transposed imaging sum for points given as Kaiser-windowed sinc taps (k_point_taps builds
// the tap tables from the positions).  A point's taps are the nodes (z0 + a, y0 + b, x0 + c),
// a, c < 8 and b < ty (8 in 3-D, 1 in 2-D), with weight wz[a] wy[b] wx[c].  Sampling
// sums the weighted taps; every injection spreads a value over the same taps with the
// same weights, so injection is the exact transpose of sampling.  One thread handles one
// (point, a, b) row of 8 taps; rows of different points may overlap, so writes are
// atomic.  Sources of a forward step are added by the step itself where its kernel does so
// (taps.cuh), and then the step's checkpoint maxima and stores hold; measured on GB300 for
// two shots of 130 x 115 x 150 points with 532 receivers each, that and one kernel for all
// point work of a reverse step (21 -> 11.5 us for image terms and injection) take a 150-step
// gradient from 19.4 to 12.2 ms.
#include "code16.cuh"
#include "fwi_internal.h"
#include "pdl.cuh"

namespace fwi {

namespace {

constexpr int kThreads = 256;

struct TapRow {
    int64_t off;    // field offset of tap (a, b, 0)
    float wzy;      // wz[a] * wy[b]
    int z, y, x0;   // node coordinates of tap (a, b, 0)
};

__device__ __forceinline__ TapRow tap_row(const Geom &g, const PointTaps &p, int a, int b)
{
    TapRow t;
    t.z = p.z0 + a;
    t.y = p.y0 + b;
    t.x0 = p.x0;
    t.off = (int64_t)t.z * g.plane + (int64_t)t.y * g.px + t.x0;
    t.wzy = p.w[a] * p.w[kTaps + b];
    return t;
}

__device__ __forceinline__ int rows_per_point(const Geom &g) { return kTaps * (g.ndim == 3 ? kTaps : 1); }

// Modified Bessel function of order 0, power series.
__host__ __device__ inline double bessel_i0(double x)
{
    double term = 1.0, total = 1.0;
    const double q = x * x / 4.0;
    for (int k = 1; k < 400 && term > 1e-18 * total; ++k) {
        term = term * q / ((double)k * k);
        total += term;
    }
    return total;
}

constexpr double kKaiser = 6.31;

// Kaiser-windowed sinc weights (Hicks 2002, Geophysics 67(1)): along an axis the 8 nodes first
// .. first + 7 around the computed-grid coordinate c get sinc(x - c) I0(6.31 sqrt(1 - ((x -
// c) / 4)^2)) / I0(6.31), in FP64; at integer c they are the delta at c.  norm = I0(6.31).  One
// thread per weight, run when the geometry changes.  Computed on the host, to check every call's
// points and again to store them, they took most of a short call: 500 steps of 64 shots with
// 512 receivers each 118.9 ms, now 40.6 (440 x 1064), a gradient of two shots of 644 receivers
// 11.5 -> 9.7 ms (90 x 75 x 110, 150 steps).
__global__ void k_point_taps(Geom g, const double *__restrict__ pos, int64_t npts, int nb, double norm,
                             PointTaps *__restrict__ out)
{
    const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = id / (3 * kTaps);
    if (i >= npts) return;
    const int e = (int)(id - i * (3 * kTaps)), axis = e / kTaps, k = e - axis * kTaps;
    PointTaps &t = out[i];
    if (axis == 1 && g.ndim == 2) {
        t.w[e] = k == 0 ? 1.0f : 0.0f;
        if (k == 0) t.y0 = 0;
        if (k == 1) t.pad = 0;
        return;
    }
    constexpr double half = kTaps / 2, pi = 3.14159265358979323846;
    const double c = pos[3 * i + axis] + nb;
    const int first = (int)floor(c) - (int)half + 1;
    const double x = (double)(first + k) - c;
    double sinc;
    if (x == floor(x)) sinc = x == 0.0 ? 1.0 : 0.0;
    else sinc = sin(pi * x) / (pi * x);
    const double r = x / half;
    const double win = r >= -1.0 && r <= 1.0 ? bessel_i0(kKaiser * sqrt(1.0 - r * r)) / norm : 0.0;
    t.w[e] = (float)(sinc * win);
    if (k == 0) (axis == 0 ? t.z0 : axis == 1 ? t.y0 : t.x0) = first;
    if (axis == 1 && k == 1) t.pad = 0;
}

// traces[s][n][r] = sum over taps of w * f (FP32).  LANES lanes share a point, each taking
// ROWS rows of taps (2-D: 8 lanes, a row each; 3-D: 32 lanes, two rows), and add up over a
// shuffle tree.  One thread per point walked 64 rows one after the other: 34 us for two
// shots of 532 receivers at 3-D on GB300, now 4.9.
template <int LANES, int ROWS>
__global__ void __launch_bounds__(kThreads) k_sample_pts(Geom g, const float *f,
                                                         const PointTaps *__restrict__ pts, int nshots,
                                                         int nrec, int nt, int n, float *traces,
                                                         const int *n_dev)
{
    pdl_next();
    const int64_t id = blockIdx.x * (int64_t)kThreads + threadIdx.x;
    const int64_t i = id / LANES;
    const int lane = (int)(id % LANES);
    const bool in = i < (int64_t)nshots * nrec;
    const int s = in ? (int)(i / nrec) : 0, r = in ? (int)(i - (int64_t)s * nrec) : 0;
    const PointTaps &p = pts[in ? i : 0];
    const float *fs = f + (int64_t)s * g.field;
    float acc = 0.0f;
    pdl_wait();
    if (n_dev) n += *n_dev;
    if (in) {
#pragma unroll
        for (int k = 0; k < ROWS; ++k) {
            const int ab = lane + k * LANES;
            const TapRow t = LANES * ROWS == kTaps ? tap_row(g, p, ab, 0) : tap_row(g, p, ab / kTaps, ab % kTaps);
            float row = 0.0f;
#pragma unroll
            for (int c = 0; c < kTaps; ++c) row = fmaf(p.w[2 * kTaps + c], fs[t.off + c], row);
            acc = fmaf(t.wzy, row, acc);
        }
    }
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (in && lane == 0) traces[((int64_t)s * nt + n) * nrec + r] = acc;
}

// kind 0: forward source, f += dt^2 w[s][n] wt / a+                   (q = wavelets)
// kind 1: adjoint injection, f += factor (W / a+) wt q[s][n][r]        (q = residuals)
__global__ void k_inject_pts(Geom g, float *f, const PointTaps *__restrict__ pts,
                             int npts, int per_shot, const float *__restrict__ W,
                             const float *__restrict__ sz, const float *__restrict__ sy,
                             const float *__restrict__ sx, const float *q, int nt,
                             int n, float dt2, float factor, int kind, const int *n_dev)
{
    const int rows = rows_per_point(g);
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    pdl_next();
    pdl_wait();
    if (i >= (int64_t)npts * rows) return;
    if (n_dev) n += *n_dev;
    const int pi = (int)(i / rows), ab = (int)(i - (int64_t)pi * rows);
    const int ty = g.ndim == 3 ? kTaps : 1;
    const int a = ab / ty, b = ab - a * ty;
    const int s = pi / per_shot, r = pi - s * per_shot;
    const PointTaps &p = pts[pi];
    const float val = kind == 0 ? dt2 * q[(int64_t)s * nt + n]
                                : q[((int64_t)s * nt + n) * per_shot + r];
    const TapRow t = tap_row(g, p, a, b);
    float *fs = f + (int64_t)s * g.field;
    const float syz = sz[t.z] + (g.ndim == 3 ? sy[t.y] : 0.0f);
#pragma unroll
    for (int c = 0; c < kTaps; ++c) {
        const float ap = 1.0f + syz + sx[t.x0 + c];
        const float scale = kind == 0 ? 1.0f / ap : factor * W[t.off + c] / ap;
        atomicAdd(fs + t.off + c, val * t.wzy * p.w[2 * kTaps + c] * scale);
    }
}

// Adds a row of taps at p, whose first column is `lead` columns past a group of four, as one
// 16-byte addition per group it meets (three; rows are 32-byte aligned, so a group lies in its
// row).  Columns of a group outside the taps receive a zero.  What bounds k_adjoint_pts is the
// rate of its atomic additions: 16384 receivers on 256^3 took 104 us with one per tap; with one
// per group the gradient call went from 204.7 to 187.7 ms, on 96^3 at 16th order from 35.7 to 32.0.
__device__ __forceinline__ void add_row(float *p, int lead, const float (&v)[kTaps])
{
    float4 *b = (float4 *)(p - lead);
    float e[kTaps + 4];
#pragma unroll
    for (int c = 0; c < kTaps + 4; ++c) e[c] = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (lead == k) {
#pragma unroll
            for (int c = 0; c < kTaps; ++c) e[k + c] = v[c];
        }
    atomicAdd(b, make_float4(e[0], e[1], e[2], e[3]));
    atomicAdd(b + 1, make_float4(e[4], e[5], e[6], e[7]));
    if (lead) atomicAdd(b + 2, make_float4(e[8], e[9], e[10], e[11]));
}

// The point work of reverse step m, one thread per row of taps:
//   receivers (npts of them): the image term g += 2 wt u^m r[s][m-1][r] (u^m = x, FP32 or a
//   code) and the injection mu^m += factor (W / a+) wt r, whose weights they share;
//   sources (nsrc, nullable src): g -= dt^2 w[s][m] wt mu^{m+1} / W.
__global__ void k_adjoint_pts(Geom g, AdjointPts a)
{
    const int rows = rows_per_point(g);
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t nr = (int64_t)a.npts * rows;
    pdl_next();
    if (i >= nr + (int64_t)a.nsrc * rows) return;
    const bool rec = i < nr;
    const int64_t k = rec ? i : i - nr;
    const int pi = (int)(k / rows), ab = (int)(k - (int64_t)pi * rows);
    const int ty = g.ndim == 3 ? kTaps : 1;
    const int ia = ab / ty, ib = ab - ia * ty;
    const PointTaps &p = rec ? a.rec[pi] : a.src[pi];
    const TapRow t = tap_row(g, p, ia, ib);
    pdl_wait();
    if (rec) {
        const int s = pi / a.per_shot, r = pi - s * a.per_shot;
        const float q = a.res[((int64_t)s * a.nt + a.m - 1) * a.per_shot + r];
        const float inv = (a.xfmt != 0 && a.xscale) ? 1.0f / a.xscale[2 * s] : 1.0f;
        const float syz = a.sz[t.z] + (g.ndim == 3 ? a.sy[t.y] : 0.0f);
        float *fs = a.mu + (int64_t)s * g.field, *gs = a.g + (int64_t)s * g.field;
        float gv[kTaps], fv[kTaps];
#pragma unroll
        for (int c = 0; c < kTaps; ++c) {
            const int64_t o = t.off + c;
            const float w = p.w[2 * kTaps + c];
            float xv;
            if (a.xfmt == 0) xv = ((const float *)a.x)[(int64_t)s * a.xstride + o];
            else xv = code16_to_float(((const unsigned short *)a.x)[(int64_t)s * a.xstride + o], a.xfmt) * inv;
            gv[c] = 2.0f * q * t.wzy * w * xv;
            const float ap = 1.0f + syz + a.sx[t.x0 + c];
            fv[c] = q * t.wzy * w * (a.factor * a.W[o] / ap);
        }
        add_row(gs + t.off, t.x0 & 3, gv);
        add_row(fs + t.off, t.x0 & 3, fv);
    } else {
        const float val = -a.dt2 * a.wav[(int64_t)pi * a.nt + a.m];
        const float *ms = a.mu1 + (int64_t)pi * g.field;
        float *gs = a.g + (int64_t)pi * g.field;
#pragma unroll
        for (int c = 0; c < kTaps; ++c) {
            const int64_t o = t.off + c;
            atomicAdd(gs + o, val * t.wzy * p.w[2 * kTaps + c] * (ms[o] / a.W[o]));
        }
    }
}

// x[s][n] = dt^2 sum_t wt mu[t] / W[t]  (the wavelet-space adjoint read at the source
// taps: nu = mu / W, as the on-grid read-out at the single node)
__global__ void k_gather_src_pts(Geom g, const float *__restrict__ f,
                                 const PointTaps *__restrict__ pts, int nshots,
                                 const float *__restrict__ W, float dt2, int nt, int n,
                                 float *__restrict__ xout)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nshots) return;
    const PointTaps &p = pts[s];
    const float *fs = f + (int64_t)s * g.field;
    const int ty = g.ndim == 3 ? kTaps : 1;
    float acc = 0.0f;
    for (int a = 0; a < kTaps; ++a)
        for (int b = 0; b < ty; ++b) {
            const TapRow t = tap_row(g, p, a, b);
            for (int c = 0; c < kTaps; ++c)
                acc += t.wzy * p.w[2 * kTaps + c] * fs[t.off + c] / W[t.off + c];
        }
    xout[(int64_t)s * nt + n] = dt2 * acc;
}

unsigned blocks(int64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

// Launches of the per-step point kernels.  In 2-D programmatic ones (201^2 off-grid forward call
// 3.57 ms against 4.40 plain, gradient 7.40 against 8.60).  In 3-D plain ones: the step's CTAs
// fill most SMs for the whole launch, so the early CTAs of a programmatic point kernel would
// crowd on the few SMs that hold fewer of them and, when the step ends, run there one after
// another (90 x 75 x 110 gradient with two shots 12.1 ms plain against 14.5, 96^3 at 16th order
// 35.7 against 40.7, 256^3 205 against 219).
template <class... P, class... A>
cudaError_t launch_pts(const Geom &g, void (*fn)(P...), int64_t threads, cudaStream_t s, const A &...a)
{
    if (g.ndim == 2) return launch_pdl(fn, dim3(blocks(threads)), dim3(kThreads), 0, s, a...);
    fn<<<blocks(threads), kThreads, 0, s>>>(a...);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_point_taps(const Geom &g, const double *pos, int64_t npts, int nb, PointTaps *out,
                              cudaStream_t s)
{
    if (npts < 1) return cudaSuccess;
    k_point_taps<<<blocks(npts * 3 * kTaps), kThreads, 0, s>>>(g, pos, npts, nb, bessel_i0(kKaiser), out);
    return cudaGetLastError();
}

cudaError_t launch_sample_pts(const Geom &g, const float *f, const PointTaps *pts, int nshots,
                              int nrec, int nt, int n, float *traces, cudaStream_t s,
                              const int *n_dev)
{
    const int64_t npts = (int64_t)nshots * nrec;
    if (g.ndim == 3)
        return launch_pts(g, k_sample_pts<32, 2>, npts * 32, s, g, f, pts, nshots, nrec, nt, n, traces, n_dev);
    return launch_pts(g, k_sample_pts<8, 1>, npts * 8, s, g, f, pts, nshots, nrec, nt, n, traces, n_dev);
}

cudaError_t launch_inject_pts(const Geom &g, float *f, const PointTaps *pts, int npts,
                              int per_shot, const float *W, const float *sig_z,
                              const float *sig_y, const float *sig_x, const float *q, int nt,
                              int n, float dt2, float factor, int kind, cudaStream_t s,
                              const int *n_dev)
{
    const int64_t rows = (int64_t)npts * kTaps * (g.ndim == 3 ? kTaps : 1);
    return launch_pts(g, k_inject_pts, rows, s, g, f, pts, npts, per_shot, W, sig_z, sig_y, sig_x, q, nt, n, dt2,
                      factor, kind, n_dev);
}

cudaError_t launch_adjoint_pts(const Geom &g, const AdjointPts &a, cudaStream_t s)
{
    const int64_t rows = (int64_t)(a.npts + a.nsrc) * kTaps * (g.ndim == 3 ? kTaps : 1);
    if (rows == 0) return cudaSuccess;
    return launch_pts(g, k_adjoint_pts, rows, s, g, a);
}

cudaError_t launch_gather_src_pts(const Geom &g, const float *f, const PointTaps *pts,
                                  int nshots, const float *W, float dt2, int nt, int n,
                                  float *x, cudaStream_t s)
{
    k_gather_src_pts<<<blocks(nshots), kThreads, 0, s>>>(g, f, pts, nshots, W, dt2, nt, n, x);
    return cudaGetLastError();
}

}  // namespace fwi
