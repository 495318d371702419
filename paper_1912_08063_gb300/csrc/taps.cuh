// An off-grid source added by a step's epilogue: the injection kernel's arithmetic (k_points.cu)
// on the 4 points of a group, so that the step's own samples, checkpoint maxima and stores see
// the injected state.
#pragma once

#include "fwi_internal.h"

namespace fwi {

// Whether rows z .. z + nz - 1, y .. y + ny - 1 of the group at column x meet the point's taps.
__device__ __forceinline__ bool taps_meet(const PointTaps &t, int dims, int z, int nz, int y, int ny, int x)
{
    const int ty = dims == 3 ? kTaps : 1;
    return z < t.z0 + kTaps && z + nz > t.z0 && y < t.y0 + ty && y + ny > t.y0 && x < t.x0 + kTaps && x + 4 > t.x0;
}

// o += val wt / a+ at the group (z, y, x .. x + 3); val = dt^2 w[n], syz the rows' damping.
__device__ __forceinline__ void add_taps(const PointTaps &t, int dims, int z, int y, int x, float val, float syz,
                                         float4 sx, float4 &o)
{
    const int a = z - t.z0, b = y - t.y0;
    if (a < 0 || a >= kTaps || b < 0 || b >= (dims == 3 ? kTaps : 1)) return;
    const float wzy = t.w[a] * t.w[kTaps + b];
    float v[4] = {o.x, o.y, o.z, o.w};
    const float s[4] = {sx.x, sx.y, sx.z, sx.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int c = x + e - t.x0;
        if (c < 0 || c >= kTaps) continue;
        const float scale = 1.0f / (1.0f + syz + s[e]);
        v[e] = __fadd_rn(v[e], __fmul_rn(__fmul_rn(__fmul_rn(val, wzy), t.w[2 * kTaps + c]), scale));
    }
    o = make_float4(v[0], v[1], v[2], v[3]);
}

}  // namespace fwi
