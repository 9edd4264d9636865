// Degridding of visibilities sorted by tile (bins.cuh).
//
// A CTA claims an item, copies the tile's region of the subgrid (39 x 39
// columns of four samples for 32 x 32 starts) into shared memory with one
// tensor copy, and its warps sum the item's visibilities four at a time: lane
// 8v + b takes row b of visibility v,
//     R_b = sum_a g_u[a] sum_c g_w[c] s[b][a][c],
// and the eight lanes of a visibility combine as in the gather kernel, two
// steps' visibilities at a time (the even lanes end with one, the odd lanes
// with the other: half the shuffles).  Every
// operation and its order match the gather and footprint-cache kernels, so
// all three agree bit for bit.  A region row is 16 bytes more than a multiple
// of 128, so the eight rows of a footprint start in eight different bank
// groups.  A lane loads the record of the visibility two steps ahead and the
// g_u and g_v rows of the next.
//
// What bounds it: 16 reads of 128 bytes from shared memory per visibility
// in complex64 (8 in FP16/BF16) at one per cycle and SM, where the gather
// kernel's 2.3 KB per visibility came from L2.  With the rows of the tables,
// the records and the shuffles it is 24 cycles per visibility, 80% of the
// data path's.  4M visibilities scattered over 16 subgrids, with the sort:
// 565 -> 380 us in complex64; 1.2M over 13 in FP16, compensated: 170 -> 124
// (391 and 129 with the shuffles of every visibility by itself).
//
// Requirements (checked by the host): as the gather kernel.
#include "bins.cuh"
#include "footprint.cuh"
#include "pipeline.cuh"
#include "tma.cuh"

namespace dg {
namespace {

constexpr int kTThreads = 256;
constexpr int kTVis = 4;                                    // visibilities per warp and step
constexpr int kRegion = (1 << kDegridTile.lx) + kUV - 1;     // columns and rows of a region
static_assert(kDegridTile.lx == kDegridTile.ly, "square tiles");

template <int DT>
struct RegionShape {
    static constexpr int kRowBytes = kRegion * kW * Storage<DT>::kBytes;
    // the smallest row of 128 k + 16 bytes
    static constexpr int kPitch = (kRowBytes - 16 + 127) / 128 * 128 + 16;
    static constexpr int kBoxX = kPitch / Storage<DT>::kBytes;
    static constexpr int kBytes = kRegion * kPitch;
    static constexpr int kSmem = (kBytes + 127) / 128 * 128;
    static constexpr int kBlocks = DT == DG_C64 ? 4 : 5;
    static_assert(kBoxX <= 256, "a box side");
};

__device__ __forceinline__ void tensor_copy_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int s, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(s), "r"(bar)
                 : "memory");
}

// What a lane needs of one visibility besides the region.
struct LaneVis {
    BinRecord r;
    float gu[kUV];
    float2 gv;              // g_v[b & ~1], g_v[b | 1]
};

__device__ __forceinline__ BinRecord load_record(const BinRecord *__restrict__ records, long long at, bool in)
{
    if (!in)
        return BinRecord{0, 0, 0, 0};
    const uint4 q = __ldg(reinterpret_cast<const uint4 *>(records + at));
    return BinRecord{q.x, q.y, q.z, q.w};
}

__device__ __forceinline__ void load_rows(LaneVis &v, const float *__restrict__ guv, int b)
{
    constexpr unsigned mask = (1u << kBinRowBits) - 1;
    const float *u = guv + (size_t)(v.r.ux & mask) * kUVRow;
    asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v.gu[0]), "=f"(v.gu[1]), "=f"(v.gu[2]), "=f"(v.gu[3]), "=f"(v.gu[4]), "=f"(v.gu[5]),
                   "=f"(v.gu[6]), "=f"(v.gu[7])
                 : "l"(u));
    v.gv = __ldg(reinterpret_cast<const float2 *>(guv + (size_t)(v.r.vy & mask) * kUVRow) + (b >> 1));
}

// Column a of the footprint row at `row`: its four samples.
template <int DT>
__device__ __forceinline__ void column(const unsigned char *row, int a, float2 (&s)[4])
{
    if constexpr (DT == DG_C64) {
        const float4 *r = reinterpret_cast<const float4 *>(row);
        const float4 p = r[2 * a], q = r[2 * a + 1];
        s[0] = make_float2(p.x, p.y);
        s[1] = make_float2(p.z, p.w);
        s[2] = make_float2(q.x, q.y);
        s[3] = make_float2(q.z, q.w);
    } else {
        const uint4 p = reinterpret_cast<const uint4 *>(row)[a];
        s[0] = Storage<DT>::cvt(p.x);
        s[1] = Storage<DT>::cvt(p.y);
        s[2] = Storage<DT>::cvt(p.z);
        s[3] = Storage<DT>::cvt(p.w);
    }
}

// This lane's row of the visibility: R_b.
template <int DT>
__device__ __forceinline__ float2 sum_row(const unsigned char *region, const LaneVis &v, const float4 &gw, int b)
{
    const int lx = v.r.ux >> kBinRowBits, ly = v.r.vy >> kBinRowBits;
    const unsigned char *row = region + (ly + b) * RegionShape<DT>::kPitch + lx * (kW * Storage<DT>::kBytes);
    float2 R = make_float2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < kUV; ++a) {
        float2 s[4];
        column<DT>(row, a, s);
        float2 m = __fmul2_rn(s[0], make_float2(gw.x, gw.x));
        m = __ffma2_rn(s[1], make_float2(gw.y, gw.y), m);
        m = __ffma2_rn(s[2], make_float2(gw.z, gw.z), m);
        m = __ffma2_rn(s[3], make_float2(gw.w, gw.w), m);
        R = a == 0 ? __fmul2_rn(m, make_float2(v.gu[0], v.gu[0])) : __ffma2_rn(m, make_float2(v.gu[a], v.gu[a]), R);
    }
    return R;
}

// The eight lanes of a visibility each have a row of it, RA of the group's
// visibility A and RB of its B: the even lanes end with A's sum, the odd ones
// with B's.  `gv`: the g_v pair of this lane's quarter, of A or B.  (Reducing
// one visibility at a time takes twice the shuffles.)
template <bool COMP>
__device__ __forceinline__ float2 sum_rows(const float2 &RA, const float2 &RB, const float2 &gv, int b)
{
    // quarter j = b >> 1: g_v[2j + 1] R_{2j + 1} + g_v[2j] R_{2j}
    const bool odd = b & 1;
    const float2 give = odd ? RA : RB, own = odd ? RB : RA;
    const float2 got = make_float2(__shfl_xor_sync(kFull, give.x, 1), __shfl_xor_sync(kFull, give.y, 1));
    const float2 Re = odd ? got : own, Ro = odd ? own : got;
    const float2 Q = __ffma2_rn(Ro, make_float2(gv.y, gv.y), __fmul2_rn(Re, make_float2(gv.x, gv.x)));
    // (Q_j + Q_{j^2}) + (Q_{j^1} + Q_{j^3})
    float2 V;
    if (COMP) {
        float2 e0, e;
        const float2 S = make_float2(two_sum(Q.x, __shfl_xor_sync(kFull, Q.x, 4), e0.x),
                                     two_sum(Q.y, __shfl_xor_sync(kFull, Q.y, 4), e0.y));
        V.x = two_sum(S.x, __shfl_xor_sync(kFull, S.x, 2), e.x);
        V.y = two_sum(S.y, __shfl_xor_sync(kFull, S.y, 2), e.y);
        e.x += e0.x + __shfl_xor_sync(kFull, e0.x, 2);
        e.y += e0.y + __shfl_xor_sync(kFull, e0.y, 2);
        V.x += e.x;
        V.y += e.y;
    } else {
        const float2 S = make_float2(Q.x + __shfl_xor_sync(kFull, Q.x, 4), Q.y + __shfl_xor_sync(kFull, Q.y, 4));
        V = make_float2(S.x + __shfl_xor_sync(kFull, S.x, 2), S.y + __shfl_xor_sync(kFull, S.y, 2));
    }
    return V;
}

template <int DT, bool COMP>
__global__ void __launch_bounds__(kTThreads, RegionShape<DT>::kBlocks)
tiled_degrid_kernel(const Geometry g, const __grid_constant__ CUtensorMap map, const Bins bins,
                    const float *__restrict__ scale, const float *__restrict__ guv, const float *__restrict__ gwt,
                    float2 *__restrict__ vis_out, DeviceStatus *__restrict__ status)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *region = smem_raw;
    __shared__ unsigned long long bar_word;
    __shared__ int claimed;
    const float4 *wtab = load_wtable(g, gwt, smem_raw + RegionShape<DT>::kSmem);
    const uint32_t bar = smem_u32(&bar_word);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int v = lane >> 3, b = lane & 7;
    constexpr int kStep = kTThreads / kWarp * kTVis;        // visibilities per step of the CTA
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbarrier_init();
    }
    pdl_wait();                         // the sorted records and the items
    const int total = *bins.n_items;
    unsigned parity = 0;
    while (true) {
        __syncthreads();                // the last item's region and claim have been read
        if (tid == 0)
            claimed = atomicAdd(bins.item_counter, 1);
        __syncthreads();
        if (claimed >= total)
            break;
        const BinItem it = bins.items[claimed];
        if (tid == 0) {
            fence_proxy_async();        // the region was read through the generic proxy
            mbar_arrive_expect_tx(bar, (unsigned)RegionShape<DT>::kBytes);
            tensor_copy_3d(smem_u32(region), &map, (it.tx << bins.tiling.lx) * kW, it.ty << bins.tiling.ly, it.s,
                           bar);
        }
        const BinRecord *recs = bins.records + it.start;
        const int at0 = warp * kTVis + v;
        LaneVis cur;
        cur.r = load_record(recs, at0, at0 < it.n);
        BinRecord next = load_record(recs, at0 + kStep, at0 + kStep < it.n);
        load_rows(cur, guv, b);
        float sc = 1.f;
        if (DT != DG_C64)
            sc = __ldg(scale + it.s);
        if (!__syncthreads_and(mbar_wait_bounded(bar, parity))) {
            if (tid == 0)
                atomicOr(&status->flags, kFlagTimeout);
            mbar_wait_bounded(bar, parity);     // (bounded) the copy in flight
            break;
        }
        parity ^= 1;
        // Sum this lane's row of the step at `at` and move on to the next.
        const auto step = [&](int at) {
            LaneVis nv;
            nv.r = next;
            next = load_record(recs, at + 2 * kStep, at + 2 * kStep < it.n);
            load_rows(nv, guv, b);
            const float4 gw = wtab ? wtab[cur.r.fw] : __ldg(reinterpret_cast<const float4 *>(gwt) + cur.r.fw);
            const float2 R = sum_row<DT>(region, cur, gw, b);
            cur = nv;
            return R;
        };
        for (int at = at0; at - v < it.n; at += 2 * kStep) {
            float2 gv = cur.gv;
            unsigned index = cur.r.index;
            const float2 RA = step(at);
            if (b & 1) {
                gv = cur.gv;
                index = cur.r.index;
            }
            float2 RB = make_float2(0.f, 0.f);
            if (at + kStep - v < it.n)      // the same in the whole warp
                RB = step(at + kStep);
            float2 V = sum_rows<COMP>(RA, RB, gv, b);
            if (DT != DG_C64)
                V = __fmul2_rn(V, make_float2(sc, sc));
            if (b < 2 && at + b * kStep < it.n)
                vis_out[index] = V;
        }
    }
}

template <int DT, bool COMP>
cudaError_t launch(degrid_plan *p, cudaStream_t st, const Bins &bins, long long max_items, const void *subgrids,
                   int n_subgrids, const float *scale, float2 *out)
{
    const size_t smem = RegionShape<DT>::kSmem + wtable_bytes_host(p->geo);
    static std::atomic<size_t> smem_table[kMaxDevices];
    cudaError_t e = dg_open_smem(dg_smem_record(smem_table, p->device), tiled_degrid_kernel<DT, COMP>, smem);
    if (e != cudaSuccess)
        return e;
    CUtensorMap map;
    e = encode_3d(&map, const_cast<void *>(subgrids),
                  DT == DG_C64 ? CU_TENSOR_MAP_DATA_TYPE_UINT64 : CU_TENSOR_MAP_DATA_TYPE_UINT32,
                  (uint64_t)p->geo.row_stride, (uint64_t)p->geo.ny, (uint64_t)n_subgrids, Storage<DT>::kBytes,
                  (uint32_t)RegionShape<DT>::kBoxX, (uint32_t)kRegion);
    if (e != cudaSuccess)
        return e;
    const long long most = (long long)p->sm_count * RegionShape<DT>::kBlocks;
    return launch_pdl(tiled_degrid_kernel<DT, COMP>, dim3((unsigned)(max_items < most ? max_items : most)),
                      dim3(kTThreads), smem, st, p->geo, map, bins, scale, (const float *)p->guv,
                      (const float *)p->gw, out, p->status);
}

}  // namespace
}  // namespace dg

cudaError_t dg_launch_tiled_degrid(degrid_plan *p, cudaStream_t st, const dg::Bins &bins, long long max_items,
                                   const void *subgrids, int n_subgrids, const float *scale, float *vis_out)
{
    using namespace dg;
    float2 *out = reinterpret_cast<float2 *>(vis_out);
    const auto run = [&](auto plain, auto comp) {
        return (p->compensated ? comp : plain)(p, st, bins, max_items, subgrids, n_subgrids, scale, out);
    };
    switch (p->dtype) {
    case DG_C64: return run(launch<DG_C64, false>, launch<DG_C64, true>);
    case DG_C32_F16: return run(launch<DG_C32_F16, false>, launch<DG_C32_F16, true>);
    case DG_C32_BF16: return run(launch<DG_C32_BF16, false>, launch<DG_C32_BF16, true>);
    }
    return cudaErrorInvalidValue;
}
