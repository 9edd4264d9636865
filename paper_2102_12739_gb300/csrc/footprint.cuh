// One footprint point, and the error-free sum, as the summing kernels share
// them (they round alike, so their results agree bit for bit).
#pragma once

#include "internal.cuh"

namespace dg {
namespace {

// sum_c g_w[c] s[e + c] for one footprint point (the entries of M).
// With `vec` (16-byte aligned subgrids, nz a multiple of the elements per
// 16 bytes, and a footprint start z0 that is one too) the four elements are
// read with 16-byte loads.
template <int DT>
__device__ __forceinline__ float2 footprint_point(const void *sub, int64_t e, const float4 &gw, bool vec)
{
    float2 s[4];
    if (vec) {
        Storage<DT>::load4(sub, e, s);
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            s[c] = Storage<DT>::load(sub, e + c);
    }
    float2 m;
    m.x = fmaf(s[3].x, gw.w, fmaf(s[2].x, gw.z, fmaf(s[1].x, gw.y, s[0].x * gw.x)));
    m.y = fmaf(s[3].y, gw.w, fmaf(s[2].y, gw.z, fmaf(s[1].y, gw.y, s[0].y * gw.x)));
    return m;
}

// Whether the footprint starting at `key` can use 16-byte loads.
template <int DT>
__device__ __forceinline__ bool vec_footprint(bool vec_ok, int key)
{
    return vec_ok && (key % Storage<DT>::kQuad) == 0;
}

// Error-free sum (Knuth's TwoSum): a + b = s + e exactly, s = fl(a + b).
__device__ __forceinline__ float two_sum(float a, float b, float &e)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

}  // namespace
}  // namespace dg
