// Auxiliary kernels: the coordinate step on its own (for bit-exact checks of
// the indices and GCF rows used by degrid.cu) and the conversion of complex64
// subgrids to the FP16 / BF16 storage with a per-subgrid scale.
#include "internal.cuh"

namespace dg {
namespace {

// Same device function as the degridding and gridding kernels use.
__global__ void coords_kernel(const Geometry g, const double *__restrict__ uvw, int64_t n_vis,
                              int *__restrict__ out, DeviceStatus *__restrict__ status)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < n_vis; i0 += stride) {
        const int64_t i = i0 + threadIdx.x;
        const bool in = i < n_vis;
        bool valid = false;
        if (in) {
            VisCoords c;
            valid = visibility_coords(__ldg(uvw + 3 * i), __ldg(uvw + 3 * i + 1),
                                      __ldg(uvw + 3 * i + 2), g, c);
            int *o = out + 6 * i;
            o[0] = valid ? c.x0 : -1;
            o[1] = valid ? c.y0 : -1;
            o[2] = valid ? c.z0 : -1;
            o[3] = valid ? c.fu : -1;
            o[4] = valid ? c.fv : -1;
            o[5] = valid ? c.fw : -1;
        }
        const unsigned bad = __ballot_sync(kFull, in && !valid);
        if ((threadIdx.x & 31) == 0 && bad)
            atomicAdd(&status->n_invalid, (unsigned long long)__popc(bad));
    }
}

// ---- FP16 / BF16 storage -------------------------------------------------------
//
// scale[s] = max |component| of subgrid s, codes = RN(component / scale[s]):
// two passes over the input, the second dependent on the first.  DRAM bounds
// both (32 subgrids of 512 x 512 x 4: 268 MB in, 134 MB out).
// A block takes one piece, so a pass is one grid of plain streaming blocks.

constexpr int kPackThreads = 256;
constexpr int kPieceComps = 8192;               // components per block: 32 KB in, 16 KB out

// Max |component| of components [lo, hi) of `src`, over the block.  The
// values are non-negative, so their IEEE bit patterns order like unsigned
// integers and an integer atomicMax finds the float maximum.
template <bool VEC>
__device__ __forceinline__ void pack_maximum(const float *__restrict__ src, int64_t lo, int64_t hi,
                                             float *__restrict__ scale)
{
    float m = 0.f;
    if (VEC) {
        const float4 *p = reinterpret_cast<const float4 *>(src);
#pragma unroll 8
        for (int64_t i = lo / 4 + threadIdx.x; i < hi / 4; i += kPackThreads) {
            const float4 v = __ldg(p + i);
            m = fmaxf(fmaxf(fmaxf(m, fabsf(v.x)), fmaxf(fabsf(v.y), fabsf(v.z))), fabsf(v.w));
        }
    } else {
        for (int64_t i = lo + threadIdx.x; i < hi; i += kPackThreads)
            m = fmaxf(m, fabsf(__ldg(src + i)));
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1)
        m = fmaxf(m, __shfl_xor_sync(kFull, m, d));
    __shared__ float warp_max[kPackThreads / kWarp];
    if ((threadIdx.x & 31) == 0)
        warp_max[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 1; k < kPackThreads / kWarp; ++k)
            m = fmaxf(m, warp_max[k]);
        atomicMax(reinterpret_cast<unsigned *>(scale), __float_as_uint(m));
    }
}

template <int DT>
__device__ __forceinline__ unsigned pack_bits(float q)
{
    return DT == DG_C32_F16 ? __half_as_ushort(__float2half_rn(q)) : __bfloat16_as_ushort(__float2bfloat16_rn(q));
}

template <int DT>
__device__ __forceinline__ unsigned pack_code(float x, float sc)
{
    return pack_bits<DT>(sc > 0.f ? __fdiv_rn(x, sc) : 0.f);
}

// RN(x / sc) from r = RN(1 / sc), by Markstein's theorem (IBM J. Res. Dev.
// 34(1), 1990): if q is within an ulp of x / sc and r is the correctly
// rounded reciprocal, q + r (x - q sc) with fused operations is the correctly
// rounded quotient.  x r is within 1.5 ulp; the first correction brings it
// within one.  Neither the quotient nor the remainders may underflow
// (quotient_floor).
__device__ __forceinline__ float quotient(float x, float sc, float r)
{
    float q = x * r;
    q = fmaf(fmaf(-q, sc, x), r, q);
    return fmaf(fmaf(-q, sc, x), r, q);
}

// The smallest |x| that `quotient` may be given with this scale (infinity: none).
__device__ __forceinline__ float quotient_floor(float sc)
{
    return sc >= 0x1p-40f && sc <= 0x1p100f ? sc * 0x1p-40f : __int_as_float(0x7f800000);
}

// Codes of components [lo, hi) of `src`.  The general division takes 10 of
// the 19 instructions per component of this pass and holds it below the DRAM
// rate; components within 2^-40 of the scale take five multiply-adds.
template <int DT, bool VEC>
__device__ __forceinline__ void pack_encode(const float *__restrict__ src, int64_t lo, int64_t hi, float sc,
                                            unsigned short *__restrict__ codes)
{
    if (VEC) {
        const float4 *p = reinterpret_cast<const float4 *>(src);
        uint2 *o = reinterpret_cast<uint2 *>(codes);
        const float r = __frcp_rn(sc), least = quotient_floor(sc);
#pragma unroll 8
        for (int64_t i = lo / 4 + threadIdx.x; i < hi / 4; i += kPackThreads) {
            const float4 v = __ldg(p + i);
            uint2 c;
            // (false for NaN and, through `least`, for scales out of range)
            if (fabsf(v.x) >= least && fabsf(v.y) >= least && fabsf(v.z) >= least && fabsf(v.w) >= least)
                c = make_uint2(pack_bits<DT>(quotient(v.x, sc, r)) | pack_bits<DT>(quotient(v.y, sc, r)) << 16,
                               pack_bits<DT>(quotient(v.z, sc, r)) | pack_bits<DT>(quotient(v.w, sc, r)) << 16);
            else
                c = make_uint2(pack_code<DT>(v.x, sc) | pack_code<DT>(v.y, sc) << 16,
                               pack_code<DT>(v.z, sc) | pack_code<DT>(v.w, sc) << 16);
            __stcs(o + i, c);
        }
    } else {
        for (int64_t i = lo + threadIdx.x; i < hi; i += kPackThreads)
            codes[i] = (unsigned short)pack_code<DT>(__ldg(src + i), sc);
    }
}

// Block (piece, s): the maximum of a piece of subgrid s into scale[s]
// (cleared before).
template <bool VEC>
__global__ void __launch_bounds__(kPackThreads)
pack_max_kernel(const float *__restrict__ in, int64_t comps, int pieces, float *__restrict__ scale)
{
    pdl_trigger();
    const int s = blockIdx.x / pieces;
    const int64_t lo = (int64_t)(blockIdx.x - s * pieces) * kPieceComps;
    const int64_t hi = lo + kPieceComps < comps ? lo + kPieceComps : comps;
    pack_maximum<VEC>(in + (int64_t)s * comps, lo, hi, scale + s);
}

// The codes of the same pieces, after the maxima.
template <int DT, bool VEC>
__global__ void __launch_bounds__(kPackThreads)
pack_encode_kernel(const float *__restrict__ in, int64_t comps, int pieces, const float *scale,
                   unsigned short *__restrict__ codes)
{
    const int s = blockIdx.x / pieces;
    const int64_t lo = (int64_t)(blockIdx.x - s * pieces) * kPieceComps;
    const int64_t hi = lo + kPieceComps < comps ? lo + kPieceComps : comps;
    pdl_wait();                                 // the maxima are complete
    pack_encode<DT, VEC>(in + (int64_t)s * comps, lo, hi, scale[s], codes + (int64_t)s * comps);
}

template <int DT, bool VEC>
cudaError_t launch_pack(cudaStream_t st, int n_subgrids, int64_t comps, const float *in, unsigned short *codes,
                        float *scale)
{
    const int64_t pieces = (comps + kPieceComps - 1) / kPieceComps;
    if (pieces > 0x7fffffff)
        return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(scale, 0, sizeof(float) * (size_t)n_subgrids, st);
    // the grid's blocks within 31 bits: normally every subgrid at once
    const int64_t most = 0x7fffffff / pieces;
    for (int64_t s0 = 0; s0 < n_subgrids && e == cudaSuccess; s0 += most) {
        const unsigned blocks = (unsigned)((most < n_subgrids - s0 ? most : n_subgrids - s0) * pieces);
        pack_max_kernel<VEC><<<blocks, kPackThreads, 0, st>>>(in + s0 * comps, comps, (int)pieces, scale + s0);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = launch_pdl(pack_encode_kernel<DT, VEC>, dim3(blocks), dim3(kPackThreads), 0, st, in + s0 * comps,
                           comps, (int)pieces, (const float *)scale + s0, codes + s0 * comps);
    }
    return e;
}

template <int DT>
cudaError_t pack(cudaStream_t st, int n_subgrids, int64_t comps, const float *in, unsigned short *codes, float *scale)
{
    // 16-byte loads and 8-byte stores: whole groups of four components per
    // subgrid, aligned buffers
    const bool vec = comps % 4 == 0 && (uintptr_t)in % 16 == 0 && (uintptr_t)codes % 8 == 0;
    if (!vec)
        return launch_pack<DT, false>(st, n_subgrids, comps, in, codes, scale);
    return launch_pack<DT, true>(st, n_subgrids, comps, in, codes, scale);
}

}  // namespace
}  // namespace dg

cudaError_t dg_launch_coords(degrid_plan *p, cudaStream_t st, const double *uvw,
                             int64_t n_vis, int32_t *coords_out)
{
    using namespace dg;
    if (n_vis == 0)
        return cudaSuccess;
    const int threads = 256;
    int64_t blocks = (n_vis + threads - 1) / threads;
    const int64_t cap = (int64_t)p->sm_count * 8;
    if (blocks > cap)
        blocks = cap;
    coords_kernel<<<(int)blocks, threads, 0, st>>>(p->geo, uvw, n_vis, coords_out, p->status);
    return cudaGetLastError();
}

cudaError_t dg_launch_pack(cudaStream_t st, dg_dtype dtype, int n_subgrids, int64_t elems,
                           const float *in, void *codes_out, float *scale_out)
{
    using namespace dg;
    if (n_subgrids == 0)
        return cudaSuccess;
    if (elems == 0)
        return cudaMemsetAsync(scale_out, 0, sizeof(float) * (size_t)n_subgrids, st);
    auto *codes = reinterpret_cast<unsigned short *>(codes_out);
    return dtype == DG_C32_F16
               ? pack<DG_C32_F16>(st, n_subgrids, 2 * elems, in, codes, scale_out)
               : pack<DG_C32_BF16>(st, n_subgrids, 2 * elems, in, codes, scale_out);
}
