// Reading checkpoint codes in place: four consecutive 16-bit codes (BF16 or FP16, the
// FWI_SNAP_* types 1 and 2) to FP32, times the reciprocal of the checkpoint's scale.
// Scales are powers of two, so the product equals code / scale exactly: the same values
// the decode kernel (k_aux.cu) writes.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cstdint>

namespace fwi {

__device__ __forceinline__ float code16_to_float(unsigned short h, int fmt)
{
    return fmt == 1 ? __bfloat162float(__ushort_as_bfloat16(h)) : __half2float(__ushort_as_half(h));
}

// One scaled value rounded to nearest even in BF16 (fmt 1) or FP16 (fmt 2): the encode
// kernel's arithmetic.
__device__ __forceinline__ unsigned short float_to_code16(float x, int fmt)
{
    return fmt == 1 ? __bfloat16_as_ushort(__float2bfloat16_rn(x)) : __half_as_ushort(__float2half_rn(x));
}

// Two values to two codes with one paired conversion (each element rounded to nearest
// even, x in the low half): the same bits as two float_to_code16 calls.
template <int FMT>
__device__ __forceinline__ unsigned pack_code2(float2 v)
{
    if constexpr (FMT == 1) {
        const __nv_bfloat162 h = __float22bfloat162_rn(v);
        return *reinterpret_cast<const unsigned *>(&h);
    } else {
        const __half2 h = __float22half2_rn(v);
        return *reinterpret_cast<const unsigned *>(&h);
    }
}

template <int FMT>
__device__ __forceinline__ float2 unpack_code2(unsigned u)
{
    if constexpr (FMT == 1) return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u));
    else return __half22float2(*reinterpret_cast<const __half2 *>(&u));
}

// Four values times the checkpoint's scale s, as codes packed little-endian.
__device__ __forceinline__ uint2 pack_code4(float4 v, int fmt, float s)
{
    const float2 s2 = make_float2(s, s);
    const float2 a = __fmul2_rn(make_float2(v.x, v.y), s2);
    const float2 b = __fmul2_rn(make_float2(v.z, v.w), s2);
    if (fmt == 1) return make_uint2(pack_code2<1>(a), pack_code2<1>(b));
    return make_uint2(pack_code2<2>(a), pack_code2<2>(b));
}

__device__ __forceinline__ float4 unpack_code4(uint2 raw, int fmt, float inv)
{
    float2 a, b;
    if (fmt == 1) {
        a = unpack_code2<1>(raw.x);
        b = unpack_code2<1>(raw.y);
    } else {
        a = unpack_code2<2>(raw.x);
        b = unpack_code2<2>(raw.y);
    }
    const float2 i2 = make_float2(inv, inv);
    a = __fmul2_rn(a, i2);
    b = __fmul2_rn(b, i2);
    return make_float4(a.x, a.y, b.x, b.y);
}

// s = 2^floor(log2(T / max)) with T = 2^texp, from the bit pattern of max (exact
// integer arithmetic); NaN for a non-finite max, 1 for an all-zero pair.
__device__ __forceinline__ float snap_scale(unsigned mb, int dtype)
{
    if (dtype == 0 || mb == 0u) return 1.0f;
    if (mb >= 0x7f800000u) return __int_as_float(0x7fc00000);
    const int texp = (dtype == 2) ? 14 : 0;
    const unsigned e = mb >> 23, mant = mb & 0x7fffffu;
    int E;
    bool frac;
    if (e > 0) {
        E = (int)e - 127;
        frac = mant != 0u;
    } else {
        E = (31 - __clz((int)mant)) - 149;
        frac = (mant & (mant - 1u)) != 0u;
    }
    int k = texp - E - (frac ? 1 : 0);
    k = max(-126, min(127, k));
    return __int_as_float((k + 127) << 23);
}

// The scales of a checkpoint that a step writes from its epilogue, from the maxima mx of the
// state it stores (the encode kernel's rule).
__device__ __forceinline__ float2 store_scales(const unsigned *mx, int shot, int dtype)
{
    return make_float2(snap_scale(mx[2 * shot], dtype), snap_scale(mx[2 * shot + 1], dtype));
}

// What one thread does for a shot of a forward step: publishes the scales of the checkpoint
// the step stores (raising *flag for a non-finite state) and clears the maxima that the next
// step raises.
__device__ __forceinline__ void store_bookkeeping(const unsigned *mx, int shot, int dtype, float *scale,
                                                  unsigned *flag, unsigned *clear)
{
    if (mx) {
        const float2 s = store_scales(mx, shot, dtype);
        scale[2 * shot] = s.x;
        scale[2 * shot + 1] = s.y;
        if (mx[2 * shot] >= 0x7f800000u) atomicOr(flag, 1u);
    }
    if (clear) clear[2 * shot] = clear[2 * shot + 1] = 0u;
}

}  // namespace fwi
