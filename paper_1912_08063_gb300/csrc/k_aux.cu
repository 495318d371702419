// Auxiliary kernels of the FWI hot path: model set-up (W = v^2 dt^2 on the padded grid),
// receiver sampling and adjoint injection, the FP64 misfit reduction (Eq. 1), the
// checkpoint codec (BF16/FP16 with a per-checkpoint power-of-two scale), the FP32 -> FP64
// gradient fold and the gradient finish (dW/dv and the fold of sponge cells).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "code16.cuh"
#include "fwi_internal.h"
#include "pdl.cuh"

namespace fwi {

namespace {

constexpr int kThreads = 256;

int blocks_for(int64_t n, int cap = 148 * 16)
{
    int64_t b = (n + kThreads - 1) / kThreads;
    if (b < 1) b = 1;
    return (int)(b > cap ? cap : b);
}

// ---------------------------------------------------------------- set-up

// W[c] = (v[clamp(c - nb)] dt)^2 on the computed grid, zero in the row padding.
// One CTA per computed row (z, y) at a time, threads along x (the row split is one 32-bit
// division per row, not two 64-bit ones per point).
__global__ void k_build_W(Geom g, int nb, int npz, int npy, int npx, const float *__restrict__ v,
                          double dt, float *__restrict__ W)
{
    const int nby = (g.ndim == 3) ? nb : 0;
    const int rows = g.nz * g.ny;
    for (int row = blockIdx.x; row < rows; row += gridDim.x) {
        const int z = row / g.ny, y = row - z * g.ny;
        const int pz = min(max(z - nb, 0), npz - 1), py = min(max(y - nby, 0), npy - 1);
        const float *vr = v + ((int64_t)pz * npy + py) * npx;
        float *wr = W + (int64_t)row * g.px;
        for (int x = threadIdx.x; x < g.px; x += blockDim.x) {
            float w = 0.0f;
            if (x < g.nx) {
                const double vv = vr[min(max(x - nb, 0), npx - 1)];
                w = (float)(vv * vv * dt * dt);
            }
            wr[x] = w;
        }
    }
}

// out[i] = factor * W / (1 + s)  (mode 0: adjoint receiver injection of W R^T q / a+)
// out[i] = factor / W            (mode 1: source read-out dt^2 mu / W)
__global__ void k_rec_scale(Geom g, const float *__restrict__ W, const float *__restrict__ sz,
                            const float *__restrict__ sy, const float *__restrict__ sx,
                            const int64_t *__restrict__ off, int count, float factor, int mode,
                            float *__restrict__ out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const int64_t o = off[i];
    const int64_t z = o / g.plane, r = o - z * g.plane;
    const int64_t y = r / g.px, x = r - y * g.px;
    const float w = W[o];
    if (mode == 0) {
        const float s = sz[z] + sy[y] + sx[x];
        out[i] = factor * w / (1.0f + s);
    } else {
        out[i] = factor / w;
    }
}

// ---------------------------------------------------------------- receivers

__global__ void k_sample(int64_t fs, const float *__restrict__ f, const int64_t *__restrict__ off,
                         int nshots, int nrec, int nt, int n, float *__restrict__ traces,
                         const int *__restrict__ n_dev)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nshots * nrec) return;
    const int s = i / nrec, r = i - s * nrec;
    if (n_dev) n += *n_dev;
    traces[((int64_t)s * nt + n) * nrec + r] = f[(int64_t)s * fs + off[i]];
}

__global__ void k_inject(int64_t fs, float *__restrict__ f, const int64_t *__restrict__ off,
                         const float *__restrict__ scale, const float *__restrict__ q,
                         int nshots, int nrec, int nt, int sample)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nshots * nrec) return;
    const int s = i / nrec, r = i - s * nrec;
    atomicAdd(f + (int64_t)s * fs + off[i], scale[i] * q[((int64_t)s * nt + sample) * nrec + r]);
}

// (double)x in integer instructions for zeros and normal numbers: the FP64 exponent is the
// FP32 one plus 1023 - 127, the fraction moves up by 29 bits.
__device__ __forceinline__ double widen(float x)
{
    const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu;
    if (e - 1u < 254u)
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))),
                                (int)(u << 29));
    if ((u << 1) == 0u) return __hiloint2double((int)u, 0);
    return (double)x;   // subnormal, infinite or NaN
}

// 2 sum_k d (d - dobs) in FP64 per (shot, receiver), with the residual rounded to FP32 exactly
// as the misfit kernel rounds it (the value injected into the adjoint).  A CTA takes 32
// receivers of a shot (one 128-byte line of a trace sample) and its 32 warps every 32nd
// sample; a fixed tree adds up.  One thread per receiver walked all samples: 167 us for 201
// receivers of 500 samples on GB300, now 23 (the FP64 unit bounds it).
constexpr int kRecX = 32, kRecY = 32;

__global__ void __launch_bounds__(kRecX * kRecY)
k_rec_image(int64_t fs, const float *__restrict__ d, const float *__restrict__ dobs,
            const int64_t *__restrict__ off, int nrec, int nt, double *__restrict__ g)
{
    __shared__ double part[kRecY][kRecX];
    const int s = blockIdx.y, r = blockIdx.x * kRecX + threadIdx.x;
    double acc = 0.0;
    if (r < nrec) {
#pragma unroll 4
        for (int k = threadIdx.y; k < nt; k += kRecY) {
            const int64_t t = ((int64_t)s * nt + k) * nrec + r;
            const float dd = d[t];
            const float rr = dd - dobs[t];
            acc = fma(widen(dd), widen(rr), acc);
        }
    }
    part[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
#pragma unroll
    for (int h = kRecY / 2; h > 0; h >>= 1) {
        if (threadIdx.y < h) part[threadIdx.y][threadIdx.x] += part[threadIdx.y + h][threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.y == 0 && r < nrec)
        atomicAdd(g + (int64_t)s * fs + off[(int64_t)s * nrec + r], 2.0 * part[0][threadIdx.x]);
}

// One thread per shot: g[src] -= dt^2 w[0] mu^1[src] / W[src], the m = 0 source term of
// the transposed imaging sum (the reverse sweep ends with the step that makes mu^1).
__global__ void k_src_image(int64_t fs, const float *__restrict__ mu1,
                            const int64_t *__restrict__ off, const float *__restrict__ W,
                            const float *__restrict__ wav, float dt2, int nshots, int nt,
                            double *__restrict__ g)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nshots) return;
    const int64_t o = off[s];
    const float f0 = dt2 * wav[(int64_t)s * nt];
    g[(int64_t)s * fs + o] -= (double)f0 * (double)mu1[(int64_t)s * fs + o] / (double)W[o];
}

__global__ void k_gather_src(int64_t fs, const float *__restrict__ f,
                             const int64_t *__restrict__ off, const float *__restrict__ sc,
                             int nshots, int nt, int sample, float *__restrict__ x)
{
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nshots) return;
    x[(int64_t)s * nt + sample] = f[(int64_t)s * fs + off[s]] * sc[s];
}

// ---------------------------------------------------------------- misfit (Eq. 1)

__device__ double block_sum(double v)
{
    __shared__ double part[kThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) part[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (wid == 0) {
        t = lane < kThreads / 32 ? part[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    return t;  // valid in thread 0
}

// Fixed-order partial sums: thread t of block b adds samples b*T + t + k*(B*T), k = 0.. in
// order, then a fixed tree.  The grid size depends only on n, so the result is
// reproducible bit for bit.
__global__ void k_misfit_partial(const float *__restrict__ d, const float *__restrict__ dobs,
                                 float *__restrict__ r_out, int64_t n, double *__restrict__ part)
{
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * kThreads) {
        const float r = d[i] - dobs[i];
        if (r_out) r_out[i] = r;
        acc += (double)r * (double)r;
    }
    const double t = block_sum(acc);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void k_sum_partials(const double *__restrict__ part, int nb, double *__restrict__ out,
                               unsigned *flag)
{
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += kThreads) acc += part[i];
    const double t = block_sum(acc);
    if (threadIdx.x == 0) {
        out[0] = t;
        if (flag && !isfinite(t)) atomicOr(flag, 1u);
    }
}

// ---------------------------------------------------------------- checkpoint codec

__device__ __forceinline__ unsigned absbits(float x) { return __float_as_uint(x) & 0x7fffffffu; }

// max(|m|, |x|) with NaN propagated; the sign of the result is not meaningful.
__device__ __forceinline__ float absmax_nan(float m, float x)
{
    float r;
    asm("max.NaN.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(m), "f"(x));
    return r;
}

// Groups of four values of a field that a codec thread loads before it uses the first: maxima,
// encode, decode.  The loads are plain (pdl.cuh), so the compiler moves none of the next round
// above a store.  26 M values on GB300, us a call, encode with 4 / 4, 8 / 1, 8 / 2, 8 / 4 (maxima /
// encode) 92.4, 88.3, 76.5, 83.6, 84.5 with non-coherent loads and 4 / 1; decode with 4 50.0, 54.4
// with non-coherent loads and 1.
constexpr int kMaxBatch = 8, kEncBatch = 2, kDecBatch = 4;

// Running maxima of |a|, |b| and |a - b|.
struct PairMax {
    float a = 0.0f, b = 0.0f, d = 0.0f;
    __device__ __forceinline__ void add(float x, float y)
    {
        a = absmax_nan(a, x);
        b = absmax_nan(b, y);
        d = absmax_nan(d, x - y);
    }
    __device__ __forceinline__ void add(float4 x, float4 y)
    {
        add(x.x, y.x);
        add(x.y, y.y);
        add(x.z, y.z);
        add(x.w, y.w);
    }
    // bits of max|a| and max|a - b| over the warp; a NaN or infinity in a or b drives both to
    // >= 0x7f800000
    __device__ __forceinline__ uint2 warp() const
    {
        const unsigned bad = absbits(a) >= 0x7f800000u || absbits(b) >= 0x7f800000u ? 0x7fc00000u : 0u;
        return make_uint2(__reduce_max_sync(0xffffffffu, max(absbits(a), bad)),
                          __reduce_max_sync(0xffffffffu, max(absbits(d), bad)));
    }
};

// out[2s] = bits of max|a|, out[2s+1] = bits of max|a - b| (FP32 difference) per shot s;
// a NaN or infinity anywhere in a or b drives both to >= 0x7f800000.  VEC reads 16 bytes a
// load, kMaxBatch loads of each field in flight (n a multiple of 4, 16-byte aligned fields), and
// a CTA joins its warps' maxima before the two atomics.
template <bool VEC>
__global__ void k_maxabs(const float *a, const float *b, int64_t n, int64_t stride, unsigned *out)
{
    const int s = blockIdx.y;
    const float *pa = a + s * stride, *pb = b + s * stride;
    PairMax m;
    pdl_next();
    pdl_wait();
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (VEC) {
        const int64_t n4 = n / 4;
        for (; i + (kMaxBatch - 1) * step < n4; i += kMaxBatch * step) {
            float4 x[kMaxBatch], y[kMaxBatch];
#pragma unroll
            for (int k = 0; k < kMaxBatch; ++k) {
                x[k] = ((const float4 *)pa)[i + k * step];
                y[k] = ((const float4 *)pb)[i + k * step];
            }
#pragma unroll
            for (int k = 0; k < kMaxBatch; ++k) m.add(x[k], y[k]);
        }
        for (; i < n4; i += step) m.add(((const float4 *)pa)[i], ((const float4 *)pb)[i]);
    } else {
        for (; i < n; i += step) m.add(pa[i], pb[i]);
    }
    __shared__ uint2 part[kThreads / 32];
    const uint2 w = m.warp();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = w;
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint2 p = threadIdx.x < kThreads / 32 ? part[threadIdx.x] : make_uint2(0u, 0u);
        const unsigned a0 = __reduce_max_sync(0xffffffffu, p.x), d0 = __reduce_max_sync(0xffffffffu, p.y);
        if (threadIdx.x == 0) {
            if (a0) atomicMax(out + 2 * s, a0);
            if (d0) atomicMax(out + 2 * s + 1, d0);
        }
    }
}

// The scales of one pair from its maxima, in place (both are two words).
__global__ void k_scales(float *scale, int dtype)
{
    pdl_next();
    pdl_wait();
    const unsigned a = __float_as_uint(scale[0]), d = __float_as_uint(scale[1]);
    scale[0] = snap_scale(a, dtype);
    scale[1] = snap_scale(d, dtype);
}

// One value of the codec: FP32 copy, or x * scale rounded to the 16-bit format.
__device__ __forceinline__ void put_code(void *code, int64_t i, int dtype, float x, float sc)
{
    if (dtype == 0) ((float *)code)[i] = x;
    else if (dtype == 1) ((__nv_bfloat16 *)code)[i] = __float2bfloat16_rn(x * sc);
    else ((__half *)code)[i] = __float2half_rn(x * sc);
}

// inv = 1 / scale.  Scales are powers of two (2^-126 .. 2^127), so their reciprocals are
// exact and code * inv equals code / scale bit for bit.
__device__ __forceinline__ float get_code(const void *code, int64_t i, int dtype, float inv)
{
    if (dtype == 0) return ((const float *)code)[i];
    if (dtype == 1) return __bfloat162float(((const __nv_bfloat16 *)code)[i]) * inv;
    return __half2float(((const __half *)code)[i]) * inv;
}

// 16-bit formats store a = u^n and d = u^n - u^{n-1}, each with its own scale; FP32
// stores the pair unchanged (lossless).  comps = 1 stores or restores a only (a
// checkpoint that is only ever restored for an imaging step, which needs u^n alone).
// VEC processes four values per thread (n a multiple of 4, 16-byte aligned fields).  The
// scales come from maxbits, which a pass over the same fields has just raised, and are
// written out; without maxbits they are read from scale (FP32 needs none: it writes 1 and
// looks for non-finite values itself).  The fields are walked from the end: what the pass
// before read last is still in L2.
template <bool VEC>
__global__ void k_encode(const float *a, const float *b, int64_t n, int64_t stride, int dtype,
                         const unsigned *maxbits, void *code, int64_t cstride, float *scale,
                         unsigned *flag, int comps)
{
    const int s = blockIdx.y;
    float sa = 1.0f, sd = 1.0f;
    pdl_next();
    pdl_wait();
    if (maxbits) {
        sa = snap_scale(maxbits[2 * s], dtype);
        sd = snap_scale(maxbits[2 * s + 1], dtype);
        if (flag && blockIdx.x == 0 && threadIdx.x == 0 && maxbits[2 * s] >= 0x7f800000u) atomicOr(flag, 1u);
    } else if (dtype != 0) {
        sa = scale[2 * s];
        sd = scale[2 * s + 1];
    }
    if ((maxbits || dtype == 0) && blockIdx.x == 0 && threadIdx.x == 0) {
        scale[2 * s] = sa;
        scale[2 * s + 1] = sd;
    }
    const bool look = !maxbits && dtype == 0 && flag;
    bool bad = false;
    const float *pa = a + s * stride, *pb = b + s * stride;
    const int esz = dtype == 0 ? 4 : 2;
    void *ca = (char *)code + (size_t)s * cstride * esz;
    void *cd = (char *)ca + (size_t)n * esz;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    if (VEC) {
        auto put = [&](int64_t i4, float4 va, float4 vb) {
            if (dtype == 0) {
                ((float4 *)ca)[i4] = va;
                if (comps == 2) ((float4 *)cd)[i4] = vb;
                if (look) {
                    PairMax m;
                    m.add(va, vb);
                    bad |= absbits(m.a) >= 0x7f800000u || absbits(m.b) >= 0x7f800000u;
                }
                return;
            }
            ((uint2 *)ca)[i4] = pack_code4(va, dtype, sa);
            if (comps == 2)
                ((uint2 *)cd)[i4] =
                    pack_code4(make_float4(va.x - vb.x, va.y - vb.y, va.z - vb.z, va.w - vb.w), dtype, sd);
        };
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const int64_t n4 = n / 4;
        int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
        for (; k + (kEncBatch - 1) * step < n4; k += kEncBatch * step) {
            float4 va[kEncBatch], vb[kEncBatch];
#pragma unroll
            for (int e = 0; e < kEncBatch; ++e) {
                const int64_t i4 = n4 - 1 - (k + e * step);
                va[e] = ((const float4 *)pa)[i4];
                vb[e] = comps == 2 ? ((const float4 *)pb)[i4] : zero4;
            }
#pragma unroll
            for (int e = 0; e < kEncBatch; ++e) put(n4 - 1 - (k + e * step), va[e], vb[e]);
        }
        for (; k < n4; k += step) {
            const int64_t i4 = n4 - 1 - k;
            put(i4, ((const float4 *)pa)[i4], comps == 2 ? ((const float4 *)pb)[i4] : zero4);
        }
    } else {
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += step) {
            const float va = pa[i];
            put_code(ca, i, dtype, va, sa);
            bad |= absbits(va) >= 0x7f800000u;
            if (comps == 2) {
                const float vb = pb[i];
                put_code(cd, i, dtype, dtype == 0 ? vb : va - vb, sd);
                bad |= absbits(vb) >= 0x7f800000u;
            }
        }
    }
    if (look && bad) atomicOr(flag, 1u);
}

// A small pair in one launch: one CTA finds the maxima, sets the scales and encodes, the
// second pass from L1 and L2.
__global__ void __launch_bounds__(1024) k_encode_small(const float *__restrict__ a, const float *__restrict__ b,
                                                       int n, int dtype, void *__restrict__ code,
                                                       float *__restrict__ scale)
{
    __shared__ uint2 part[32];
    __shared__ float2 sc;
    PairMax m;
    for (int i = threadIdx.x; i < n; i += 1024) m.add(a[i], b[i]);
    const uint2 w = m.warp();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = w;
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint2 p = part[threadIdx.x];
        const unsigned ma = __reduce_max_sync(0xffffffffu, p.x), md = __reduce_max_sync(0xffffffffu, p.y);
        if (threadIdx.x == 0) {
            sc = make_float2(snap_scale(ma, dtype), snap_scale(md, dtype));
            scale[0] = sc.x;
            scale[1] = sc.y;
        }
    }
    __syncthreads();
    void *cd = (char *)code + (size_t)n * 2;
    for (int i = threadIdx.x; i < n; i += 1024) {
        const float x = a[i], y = b[i];
        put_code(code, i, dtype, x, sc.x);
        put_code(cd, i, dtype, x - y, sc.y);
    }
}

template <bool VEC>
__global__ void k_decode(const void *code, int64_t cstride, const float *scale, int64_t n,
                         int64_t stride, int dtype, float *a, float *b, int comps)
{
    const int s = blockIdx.y;
    pdl_next();
    pdl_wait();
    const float sa = 1.0f / scale[2 * s], sd = 1.0f / scale[2 * s + 1];   // exact: powers of 2
    float *pa = a + s * stride, *pb = b + s * stride;
    const int esz = dtype == 0 ? 4 : 2;
    const void *ca = (const char *)code + (size_t)s * cstride * esz;
    const void *cd = (const char *)ca + (size_t)n * esz;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    if (VEC) {
        auto put = [&](int64_t i4, ushort4 ua, ushort4 ud) {
            const unsigned short ha[4] = {ua.x, ua.y, ua.z, ua.w};
            float xa[4], xb[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                xa[e] = (dtype == 1 ? __bfloat162float(__ushort_as_bfloat16(ha[e]))
                                    : __half2float(__ushort_as_half(ha[e]))) * sa;
            ((float4 *)pa)[i4] = make_float4(xa[0], xa[1], xa[2], xa[3]);
            if (comps == 2) {
                const unsigned short hd[4] = {ud.x, ud.y, ud.z, ud.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    xb[e] = xa[e] - (dtype == 1 ? __bfloat162float(__ushort_as_bfloat16(hd[e]))
                                                : __half2float(__ushort_as_half(hd[e]))) * sd;
                ((float4 *)pb)[i4] = make_float4(xb[0], xb[1], xb[2], xb[3]);
            }
        };
        const int64_t n4 = n / 4;
        int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
        if (dtype == 0) {
            for (; k < n4; k += step) {
                ((float4 *)pa)[k] = ((const float4 *)ca)[k];
                if (comps == 2) ((float4 *)pb)[k] = ((const float4 *)cd)[k];
            }
            return;
        }
        const ushort4 zero4 = make_ushort4(0, 0, 0, 0);
        for (; k + (kDecBatch - 1) * step < n4; k += kDecBatch * step) {
            ushort4 ua[kDecBatch], ud[kDecBatch];
#pragma unroll
            for (int e = 0; e < kDecBatch; ++e) {
                ua[e] = ((const ushort4 *)ca)[k + e * step];
                ud[e] = comps == 2 ? ((const ushort4 *)cd)[k + e * step] : zero4;
            }
#pragma unroll
            for (int e = 0; e < kDecBatch; ++e) put(k + e * step, ua[e], ud[e]);
        }
        for (; k < n4; k += step)
            put(k, ((const ushort4 *)ca)[k], comps == 2 ? ((const ushort4 *)cd)[k] : zero4);
    } else {
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += step) {
            const float va = get_code(ca, i, dtype, sa);
            pa[i] = va;
            if (comps == 2) {
                const float v = get_code(cd, i, dtype, sd);
                pb[i] = dtype == 0 ? v : va - v;
            }
        }
    }
}

__global__ void k_nonfinite(const float *__restrict__ a, int64_t n, unsigned *flag)
{
    unsigned bad = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        bad |= absbits(a[i]) >= 0x7f800000u;
    bad = __reduce_or_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && bad) atomicOr(flag, 1u);
}

// ---------------------------------------------------------------- gradient

__global__ void k_fold(float *__restrict__ g32, double *__restrict__ g64, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        g64[i] += (double)g32[i];
        g32[i] = 0.0f;
    }
}

// 1 / v for FP32 v as the sum of three FP32 terms, each from the residual 1 - v (sum so far)
// that one FMA gives (the first exactly, the second to FP32): the terms leave a relative error
// below 2^-68, under FP64's rounding.  v
// outside 2^-60 .. 2^60 takes the FP64 division (its residuals could underflow).
__device__ __forceinline__ double recip(float v)
{
    if (!(v > 8.6736174e-19f && v < 1.1529215e18f)) return 1.0 / (double)v;
    const float a = __frcp_rn(v);
    const float ra = fmaf(-v, a, 1.0f), b = ra * a;
    const float rb = fmaf(-v, b, ra), c = rb * a;
    return widen(a) + (widen(b) + widen(c));
}

// Row `i` of k_finish's two launches: rows away from the folded faces, or on them.  Faces are
// pz = 0 and npz - 1 and, in 3-D, py = 0 and npy - 1.
__host__ __device__ inline int finish_inner(int n) { return n > 2 ? n - 2 : 0; }

template <bool EDGE>
__device__ __forceinline__ void finish_row(int i, int npz, int npy, bool fold_y, int &pz, int &py)
{
    const int iy = fold_y ? finish_inner(npy) : npy;   // rows per plane away from the faces
    if (!EDGE) {
        pz = 1 + i / iy;
        py = (fold_y ? 1 : 0) + i % iy;
        return;
    }
    const int zf = npz > 1 ? 2 : 1;                     // z faces: all their rows
    if (i < zf * npy) {
        pz = i / npy == 0 ? 0 : npz - 1;
        py = i % npy;
        return;
    }
    i -= zf * npy;                                      // y faces of the planes between
    const int yf = npy > 1 ? 2 : 1;
    pz = 1 + i / yf;
    py = i % yf == 0 ? 0 : npy - 1;
}

// grad(p) = (2 / v(p)) * sum_shots sum_{computed cells c replicated from p} g_mu(c),
// where g_mu = sum_m mu^{m+1} L u^m and mu = W nu (so dphi/dW = g_mu / W and
// dphi/dv = 2 v dt^2 dphi/dW = 2 g_mu / v); g_mu is the FP64 accumulator plus the FP32
// partial since its last fold, so no separate last fold rewrites both.
//
// Bound by HBM: 12 bytes per computed cell and shot.  The sponge makes the work uneven: a
// cell on a face gathers nb + 1 cells, one on an edge (nb + 1)^2, a corner (nb + 1)^3, times
// the shots.  Rows (pz, py) away from the z and y faces (EDGE = false) and rows on them run
// as two launches; a CTA takes 256 / PARTS columns of one row and PARTS groups of threads
// share a column's list of (shot, cz, cy).  The first and last column, which also gather
// along x, are summed by a warp (PARTS = 1) or by the whole CTA.  PARTS = 1 streams rows
// whose list is the shots alone; 8 splits longer lists.  Measured on GB300 against one
// thread per cell walking its whole list after a separate fold: 64 shots of 440 x 1064
// 5128 -> 389 us, 296^3 2335 -> 551 us, 136^3 955 -> 113 us (both launches).
//
// The FP64 unit (about one operation per clock and SM) is what bounds it then, so FP32
// values are widened with integer instructions (widen) and 1 / v is built from three FP32
// terms instead of an FP64 division: 296^3 rows off the faces 1057 -> 431 us.
template <int PARTS, bool EDGE>
__global__ void __launch_bounds__(kThreads) k_finish(Geom g, int nb, int npz, int npy, int npx,
                                                     int nshots, const float *__restrict__ g32,
                                                     const double *__restrict__ g64,
                                                     const float *__restrict__ v,
                                                     float *__restrict__ grad32,
                                                     double *__restrict__ grad64, int rows, int chunks)
{
    constexpr int COLS = kThreads / PARTS;
    __shared__ double red[PARTS > 1 ? PARTS : 1][COLS];
    const bool fold_y = g.ndim == 3;
    const int nby = fold_y ? nb : 0;
    const int lane = threadIdx.x % COLS, part = threadIdx.x / COLS;
    for (int64_t w = blockIdx.x; w < (int64_t)rows * chunks; w += gridDim.x) {
        const int row = (int)(w / chunks), chunk = (int)(w - (int64_t)row * chunks);
        int pz, py;
        finish_row<EDGE>(row, npz, npy, fold_y, pz, py);
        const int z0 = pz == 0 ? 0 : pz + nb, z1 = pz == npz - 1 ? pz + 2 * nb : pz + nb;
        const int y0 = py == 0 ? 0 : py + nby, y1 = py == npy - 1 ? py + 2 * nby : py + nby;
        const int ylen = y1 - y0 + 1, zy = (z1 - z0 + 1) * ylen, list = zy * nshots;
        auto cell_row = [&](int e) {   // offset of row e of the list
            const int s = e / zy, r = e - s * zy, cz = r / ylen;
            return (int64_t)s * g.field + (int64_t)(z0 + cz) * g.plane +
                   (int64_t)(y0 + r - cz * ylen) * g.px;
        };
        auto put = [&](int pxx, double acc) {
            const int64_t i = ((int64_t)pz * npy + py) * npx + pxx;
            const double out = acc * (2.0 * recip(v[i]));
            if (grad32) grad32[i] = (float)out;
            if (grad64) grad64[i] = out;
        };
        const int pxx = chunk * COLS + lane;
        double acc = 0.0;
        if (pxx > 0 && pxx < npx - 1) {
#pragma unroll 4
            for (int e = part; e < list; e += PARTS) {
                const int64_t o = cell_row(e) + pxx + nb;
                acc += g64[o] + widen(g32[o]);
            }
        }
        if (PARTS > 1) {
            red[part][lane] = acc;
            __syncthreads();
            if (part == 0) {
#pragma unroll
                for (int k = 1; k < PARTS; ++k) acc += red[k][lane];
            }
            __syncthreads();
        }
        if (part == 0 && pxx > 0 && pxx < npx - 1) put(pxx, acc);
        // the first and the last column of the row
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const int ec = side == 0 ? 0 : npx - 1;
            if (ec / COLS != chunk || (side == 1 && npx == 1)) continue;   // uniform per CTA
            const int x0 = ec == 0 ? 0 : ec + nb, x1 = ec == npx - 1 ? ec + 2 * nb : ec + nb;
            const int xl = x1 - x0 + 1;
            const int64_t cells = (int64_t)list * xl;
            if (PARTS == 1 && (int)(threadIdx.x >> 5) != side) continue;   // one warp each
            const int64_t first = PARTS == 1 ? (threadIdx.x & 31) : threadIdx.x;
            double t = 0.0;
#pragma unroll 4
            for (int64_t c = first; c < cells; c += PARTS == 1 ? 32 : kThreads) {
                const int e = (int)(c / xl);
                const int64_t o = cell_row(e) + x0 + (int)(c - (int64_t)e * xl);
                t += g64[o] + widen(g32[o]);
            }
            if (PARTS == 1) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            } else {
                t = block_sum(t);
                __syncthreads();   // block_sum's shared words are free for the next use
            }
            if (first == 0) put(ec, t);
        }
    }
}

}  // namespace

// ---------------------------------------------------------------- launchers

cudaError_t launch_build_W(const Geom &g, int nb, const int64_t np[3], const float *v,
                           float dt, float *W, cudaStream_t s)
{
    const int rows = g.nz * g.ny;
    k_build_W<<<rows < 152 * 16 ? rows : 152 * 16, kThreads, 0, s>>>(g, nb, (int)np[0], (int)np[1],
                                                                     (int)np[2], v, dt, W);
    return cudaGetLastError();
}

__global__ void k_tick(int *counter, int add, int set)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) *counter = set ? add : *counter + add;
}

cudaError_t launch_tick(int *counter, int add, cudaStream_t s)
{
    k_tick<<<1, 32, 0, s>>>(counter, add, 0);
    return cudaGetLastError();
}

cudaError_t launch_set_counter(int *counter, int value, cudaStream_t s)
{
    k_tick<<<1, 32, 0, s>>>(counter, value, 1);
    return cudaGetLastError();
}

cudaError_t launch_sample(const Geom &g, const float *field, const int64_t *rec_off,
                          int nshots, int nrec, int nt, int n, float *traces, cudaStream_t s,
                          const int *n_dev)
{
    int cnt = nshots * nrec;
    k_sample<<<(cnt + kThreads - 1) / kThreads, kThreads, 0, s>>>(g.field, field, rec_off,
                                                                 nshots, nrec, nt, n, traces,
                                                                 n_dev);
    return cudaGetLastError();
}

cudaError_t launch_inject(const Geom &g, float *field, const int64_t *rec_off,
                          const float *scale, const float *q, int nshots, int nrec, int nt,
                          int sample, cudaStream_t s)
{
    int cnt = nshots * nrec;
    k_inject<<<(cnt + kThreads - 1) / kThreads, kThreads, 0, s>>>(g.field, field, rec_off,
                                                                 scale, q, nshots, nrec, nt,
                                                                 sample);
    return cudaGetLastError();
}

cudaError_t launch_rec_image(const Geom &g, const float *d, const float *dobs,
                             const int64_t *rec_off, int nshots, int nrec, int nt,
                             double *gacc64, cudaStream_t s)
{
    if (nshots <= 0 || nrec <= 0 || nt <= 0) return cudaSuccess;
    // shots on grid.y, at most 65535 a launch
    for (int s0 = 0; s0 < nshots; s0 += 65535) {
        const dim3 grid((nrec + kRecX - 1) / kRecX, nshots - s0 < 65535 ? nshots - s0 : 65535);
        const int64_t t0 = (int64_t)s0 * nt * nrec;
        k_rec_image<<<grid, dim3(kRecX, kRecY), 0, s>>>(g.field, d + t0, dobs + t0, rec_off + (int64_t)s0 * nrec,
                                                        nrec, nt, gacc64 + (int64_t)s0 * g.field);
    }
    return cudaGetLastError();
}

cudaError_t launch_src_image(const Geom &g, const float *mu1, const int64_t *src_off,
                             const float *W, const float *wavelet, float dt2, int nshots,
                             int nt, double *gacc64, cudaStream_t s)
{
    if (nshots <= 0) return cudaSuccess;
    k_src_image<<<(nshots + kThreads - 1) / kThreads, kThreads, 0, s>>>(
        g.field, mu1, src_off, W, wavelet, dt2, nshots, nt, gacc64);
    return cudaGetLastError();
}

cudaError_t launch_gather_src(const Geom &g, const float *field, const int64_t *src_off,
                              const float *src_scale, int nshots, int nt, int sample,
                              float *x, cudaStream_t s)
{
    k_gather_src<<<(nshots + 63) / 64, 64, 0, s>>>(g.field, field, src_off, src_scale, nshots,
                                                   nt, sample, x);
    return cudaGetLastError();
}

cudaError_t launch_rec_scale(const Geom &g, const float *W, const float *sig_z,
                             const float *sig_y, const float *sig_x, const int64_t *off,
                             int count, float factor, int mode, float *out, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    k_rec_scale<<<(count + kThreads - 1) / kThreads, kThreads, 0, s>>>(g, W, sig_z, sig_y,
                                                                      sig_x, off, count,
                                                                      factor, mode, out);
    return cudaGetLastError();
}

int misfit_blocks(int64_t n) { return blocks_for(n, 1024); }

cudaError_t launch_misfit(const float *d, const float *dobs, float *r_out, int64_t n,
                          double *partials, int nblocks, double *result, unsigned *flag,
                          cudaStream_t s)
{
    k_misfit_partial<<<nblocks, kThreads, 0, s>>>(d, dobs, r_out, n, partials);
    k_sum_partials<<<1, kThreads, 0, s>>>(partials, nblocks, result, flag);
    return cudaGetLastError();
}

static bool vec_ok(int64_t n, int64_t stride, int64_t code_stride, const void *x, const void *y,
                   const void *code)
{
    auto al = [](const void *p, int k) { return ((uintptr_t)p % k) == 0; };
    return n % 4 == 0 && stride % 4 == 0 && code_stride % 4 == 0 && al(x, 16) && al(y, 16) &&
           al(code, 16);
}

cudaError_t launch_maxabs(const float *a, const float *b, int64_t n, int64_t stride,
                          int nshots, unsigned *maxbits, cudaStream_t s)
{
    if (vec_ok(n, stride, 0, a, b, nullptr)) {
        dim3 grid(blocks_for(n / 16, 152 * 4), nshots);   // one wave
        return launch_pdl(k_maxabs<true>, grid, dim3(kThreads), 0, s, a, b, n, stride, maxbits);
    } else {
        dim3 grid(blocks_for(n, 152 * 8), nshots);
        return launch_pdl(k_maxabs<false>, grid, dim3(kThreads), 0, s, a, b, n, stride, maxbits);
    }
}

cudaError_t launch_encode_pair(const float *a, const float *b, int64_t n, int dtype, void *code,
                               float *scale, cudaStream_t s)
{
    if (dtype == 0) return launch_encode(a, b, n, n, 1, dtype, nullptr, code, 2 * n, scale, nullptr, 2, s);
    // one CTA up to 2^15 values (measured on GB300, us a call from Python, which alone takes 9:
    // 2,000 and 32,768 values 9.1 against 13.9 in four launches, 65,536 13.9 against 14.0)
    if (n <= 32768) {
        k_encode_small<<<1, 1024, 0, s>>>(a, b, (int)n, dtype, code, scale);
        return cudaGetLastError();
    }
    // the maxima gather in the two words of scale, which the caller gets back as the scales
    cudaError_t e = cudaMemsetAsync(scale, 0, 2 * sizeof(float), s);
    if (e == cudaSuccess) e = launch_maxabs(a, b, n, n, 1, (unsigned *)scale, s);
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_scales, dim3(1), dim3(1), 0, s, scale, dtype);
    if (e != cudaSuccess) return e;
    return launch_encode(a, b, n, n, 1, dtype, nullptr, code, 2 * n, scale, nullptr, 2, s);
}

cudaError_t launch_encode(const float *a, const float *b, int64_t n, int64_t stride,
                          int nshots, int dtype, const unsigned *maxbits, void *code,
                          int64_t code_stride, float *scale, unsigned *flag, int comps,
                          cudaStream_t s)
{
    if (vec_ok(n, stride, code_stride, a, b, code)) {
        dim3 grid(blocks_for(n / 4, 152 * 8), nshots);
        return launch_pdl(k_encode<true>, grid, dim3(kThreads), 0, s, a, b, n, stride, dtype, maxbits, code,
                          code_stride, scale, flag, comps);
    } else {
        dim3 grid(blocks_for(n, 152 * 8), nshots);
        return launch_pdl(k_encode<false>, grid, dim3(kThreads), 0, s, a, b, n, stride, dtype, maxbits, code,
                          code_stride, scale, flag, comps);
    }
}

cudaError_t launch_decode(const void *code, int64_t code_stride, const float *scale,
                          int64_t n, int64_t stride, int nshots, int dtype, float *a, float *b,
                          int comps, cudaStream_t s)
{
    if (vec_ok(n, stride, code_stride, a, b, code)) {
        dim3 grid(blocks_for(n / 4, 152 * 8), nshots);
        return launch_pdl(k_decode<true>, grid, dim3(kThreads), 0, s, code, code_stride, scale, n, stride, dtype,
                          a, b, comps);
    } else {
        dim3 grid(blocks_for(n, 152 * 8), nshots);
        return launch_pdl(k_decode<false>, grid, dim3(kThreads), 0, s, code, code_stride, scale, n, stride, dtype,
                          a, b, comps);
    }
}

cudaError_t launch_fold(float *g32, double *g64, int64_t n, cudaStream_t s)
{
    k_fold<<<blocks_for(n, 152 * 8), kThreads, 0, s>>>(g32, g64, n);
    return cudaGetLastError();
}

cudaError_t launch_finish(const Geom &g, int nb, const int64_t np[3], int nshots,
                          const float *g32, const double *g64, const float *v, float *grad32,
                          double *grad64, cudaStream_t s)
{
    const int npz = (int)np[0], npy = (int)np[1], npx = (int)np[2];
    const bool fold_y = g.ndim == 3;
    const int inner = finish_inner(npz) * (fold_y ? finish_inner(npy) : npy);
    const int edge = npz * npy - inner;
    auto go = [&](auto kernel, int parts, int rows) {
        if (rows < 1) return;
        const int cols = kThreads / parts, chunks = (npx + cols - 1) / cols;
        const int64_t work = (int64_t)rows * chunks;
        kernel<<<(unsigned)(work < 152 * 32 ? work : 152 * 32), kThreads, 0, s>>>(
            g, nb, npz, npy, npx, nshots, g32, g64, v, grad32, grad64, rows, chunks);
    };
    go(k_finish<8, true>, 8, edge);
    if (nshots >= 8) go(k_finish<8, false>, 8, inner);
    else go(k_finish<1, false>, 1, inner);
    return cudaGetLastError();
}

cudaError_t launch_nonfinite_check(const float *a, int64_t n, unsigned *flag, cudaStream_t s)
{
    k_nonfinite<<<blocks_for(n, 152 * 4), kThreads, 0, s>>>(a, n, flag);
    return cudaGetLastError();
}

}  // namespace fwi
