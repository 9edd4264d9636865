// Gridding of visibilities sorted by tile (bins.cuh).
//
// A warp claims an item, keeps the tile's region of the subgrid (23 x 23
// columns of four samples for 16 x 16 starts, FP32) in shared memory as a sum
// from zero, adds the item's visibilities to it one after the other, and adds
// the region to the stack with one tensor reduce-add.  The region is the
// warp's own, so the adds in it need no atomics.  For a visibility lane
// 8r + a takes column a of rows 2r and 2r + 1,
//     region[b][a][c] += g_w[c] (g_u[a] (y g_v[b])),
// as two reads and writes of 16 bytes per row.  Lanes 4 to 7 of a row take
// the upper half of their column first, so the eight lanes of a row read
// eight different bank groups.
//
// What bounds it: the 2 KB read and 2 KB written in shared memory per
// visibility, 32 accesses of 128 bytes at one per cycle and SM, where the
// scatter kernel's reduce-adds of single footprints ran at the 6.5 TB/s the
// copy engines add into L2.  2M visibilities scattered over 16 subgrids, with
// the sort and the zeros: 698 -> 391 us.  Tiles of 8 x 8 (28 warps), 8 x 16
// and 16 x 8 (20) measured 458, 407 and 406: the adds of the regions grow.
//
// Requirements (checked by the host): as the scatter kernel.
#include "bins.cuh"
#include "pipeline.cuh"
#include "tma.cuh"

namespace dg {
namespace {

constexpr int kGWarps = 12;                                 // warps per CTA (one CTA per SM)
constexpr int kGCols = (1 << kGridTile.lx) + kUV - 1;       // columns of a region
constexpr int kGRows = (1 << kGridTile.ly) + kUV - 1;       // rows
constexpr int kAhead = 4;                                   // visibilities loaded ahead
constexpr int kGPitch = kGCols * kW;                        // float2 per region row
constexpr int kGSlot = (kGRows * kGPitch * 8 + 127) / 128 * 128;      // bytes per warp

__device__ __forceinline__ void reduce_add_3d(const CUtensorMap *map, uint32_t src, int x, int y, int s)
{
    asm volatile("cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group"
                 " [%0, {%1, %2, %3}], [%4];"
                 ::"l"(map), "r"(x), "r"(y), "r"(s), "r"(src)
                 : "memory");
}

// What a lane needs of one visibility: place, y, g_u[a], g_v[2r], g_v[2r + 1]
// and the w row.
struct GridVis {
    int place;              // float4 index of column a of row 2r in the region
    unsigned fw;
    float gu;
    float2 gv, y;
};

__device__ __forceinline__ BinRecord load_record(const BinRecord *__restrict__ records, int at, int n)
{
    const uint4 q = __ldg(reinterpret_cast<const uint4 *>(records + (at < n ? at : n - 1)));
    return BinRecord{q.x, q.y, q.z, q.w};
}

__device__ __forceinline__ GridVis load_vis(const BinRecord &rec, const float *__restrict__ guv,
                                            const float2 *__restrict__ vis, int r, int a)
{
    constexpr unsigned mask = (1u << kBinRowBits) - 1;
    GridVis v;
    v.place = ((int)(rec.vy >> kBinRowBits) + 2 * r) * (kGPitch / 2) + ((int)(rec.ux >> kBinRowBits) + a) * 2;
    v.fw = rec.fw;
    v.gu = __ldg(guv + (size_t)(rec.ux & mask) * kUVRow + a);
    v.gv = __ldg(reinterpret_cast<const float2 *>(guv + (size_t)(rec.vy & mask) * kUVRow) + r);
    v.y = __ldg(vis + rec.index);
    return v;
}

__device__ __forceinline__ void add_pair(float4 &m, float2 t, float g0, float g1)
{
    const float2 p = __ffma2_rn(t, make_float2(g0, g0), make_float2(m.x, m.y));
    const float2 q = __ffma2_rn(t, make_float2(g1, g1), make_float2(m.z, m.w));
    m = make_float4(p.x, p.y, q.x, q.y);
}

// Adds a visibility to the region; `first`: which half of its column this
// lane takes first.
__device__ __forceinline__ void add_visibility(float4 *region, const GridVis &v, const float4 *wtab,
                                               const float *__restrict__ gwt, int first)
{
    const float4 gw = wtab ? wtab[v.fw] : __ldg(reinterpret_cast<const float4 *>(gwt) + v.fw);
    float4 *p0 = region + v.place + first, *p1 = region + v.place + (first ^ 1);
    float4 m0 = p0[0], m1 = p1[0], m2 = p0[kGPitch / 2], m3 = p1[kGPitch / 2];
    const float g0 = first ? gw.z : gw.x, g1 = first ? gw.w : gw.y;         // weights of p0's planes
    const float g2 = first ? gw.x : gw.z, g3 = first ? gw.y : gw.w;
    const float2 gu = make_float2(v.gu, v.gu);
    const float2 t0 = __fmul2_rn(gu, __fmul2_rn(v.y, make_float2(v.gv.x, v.gv.x)));
    const float2 t1 = __fmul2_rn(gu, __fmul2_rn(v.y, make_float2(v.gv.y, v.gv.y)));
    add_pair(m0, t0, g0, g1);
    add_pair(m1, t0, g2, g3);
    add_pair(m2, t1, g0, g1);
    add_pair(m3, t1, g2, g3);
    p0[0] = m0;
    p1[0] = m1;
    p0[kGPitch / 2] = m2;
    p1[kGPitch / 2] = m3;
}

__global__ void __launch_bounds__(kGWarps * kWarp, 1)
tiled_grid_kernel(const Geometry g, const __grid_constant__ CUtensorMap map, const Bins bins,
                  const float2 *__restrict__ vis_in, const float *__restrict__ guv, const float *__restrict__ gwt)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float4 *region = reinterpret_cast<float4 *>(smem_raw + (threadIdx.x >> 5) * kGSlot);
    const float4 *wtab = load_wtable(g, gwt, smem_raw + kGWarps * kGSlot);
    const int lane = threadIdx.x & 31, r = lane >> 3, a = lane & 7, first = (a >> 2) & 1;
    pdl_wait();                         // the sorted records, the items and the zeroed output
    const int total = *bins.n_items;
    int k = 0;
    if (lane == 0)
        k = atomicAdd(bins.item_counter, 1);
    k = __shfl_sync(kFull, k, 0);
    while (k < total) {
        const BinItem it = bins.items[k];
        int ahead = 0;
        if (lane == 0)
            ahead = atomicAdd(bins.item_counter, 1);
        const BinRecord *recs = bins.records + it.start;
        // four visibilities at a time: their rows and values loaded four
        // ahead, their records eight
        GridVis cur[kAhead];
        BinRecord next[kAhead];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            cur[q] = load_vis(load_record(recs, q, it.n), guv, vis_in, r, a);
            next[q] = load_record(recs, kAhead + q, it.n);
        }
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // lane 0: the last region has been added
        __syncwarp();
        for (int i = lane; i < kGRows * kGPitch / 2; i += kWarp)
            region[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();
        for (int i = 0; i < it.n; i += kAhead) {
            GridVis nv[kAhead];
#pragma unroll
            for (int q = 0; q < kAhead; ++q) {
                nv[q] = load_vis(next[q], guv, vis_in, r, a);
                next[q] = load_record(recs, i + 2 * kAhead + q, it.n);
            }
#pragma unroll
            for (int q = 0; q < kAhead; ++q) {
                if (i + q < it.n)
                    add_visibility(region, cur[q], wtab, gwt, first);
                __syncwarp();           // the next footprint may overlap this one
                cur[q] = nv[q];
            }
        }
        fence_proxy_async();            // the region, written by the generic proxy, goes to the copy engine
        __syncwarp();
        if (lane == 0) {
            reduce_add_3d(&map, smem_u32(region), (it.tx << bins.tiling.lx) * (kW * 2), it.ty << bins.tiling.ly, it.s);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        k = __shfl_sync(kFull, ahead, 0);
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");       // every reduce has finished before the warp ends
}

}  // namespace
}  // namespace dg

cudaError_t dg_launch_tiled_grid(degrid_plan *p, cudaStream_t st, const dg::Bins &bins, long long max_items,
                                 int n_subgrids, const float *vis_in, float *sub_out)
{
    using namespace dg;
    const size_t smem = (size_t)kGWarps * kGSlot + wtable_bytes_host(p->geo);
    static std::atomic<size_t> smem_table[kMaxDevices];
    cudaError_t e = dg_open_smem(dg_smem_record(smem_table, p->device), tiled_grid_kernel, smem);
    if (e != cudaSuccess)
        return e;
    CUtensorMap map;
    e = encode_3d(&map, sub_out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2 * (uint64_t)p->geo.row_stride,
                  (uint64_t)p->geo.ny, (uint64_t)n_subgrids, 4, (uint32_t)(2 * kGPitch), (uint32_t)kGRows);
    if (e != cudaSuccess)
        return e;
    const long long useful = (max_items + kGWarps - 1) / kGWarps;
    return launch_pdl(tiled_grid_kernel, dim3((unsigned)(useful < p->sm_count ? useful : p->sm_count)),
                      dim3(kGWarps * kWarp), smem, st, p->geo, map, bins, reinterpret_cast<const float2 *>(vis_in),
                      (const float *)p->guv, (const float *)p->gw);
}
