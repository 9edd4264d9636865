// Sorting the visibilities of a call by tile (bins.cuh): counts per tile,
// places, and the records at their places.
//
// A subgrid's records take the places of its list, [vis_offsets[s],
// vis_offsets[s + 1]), so the scan over its tiles is its own and no global
// one is needed; invalid visibilities leave a gap at the end.  A block takes
// kPiece consecutive visibilities and counts them in shared memory, so the
// global counters see one atomic per block and tile (one per visibility
// serialised on a few lines of L2: 114 us a pass for 4M visibilities over 256
// tiles per subgrid, 30 this way).  The coordinates are read and snapped in
// both passes: 24 bytes, against 16 written and read again.
#include "bins.cuh"

#include <new>

namespace dg {
namespace {

constexpr int kBinThreads = 256;
constexpr int kPiece = 1024;                // visibilities per block (512, 2048 and 4096 measured slower)
constexpr int kPerThread = kPiece / kBinThreads;
constexpr int kTilesThreads = 1024;         // most threads of bin_tiles_kernel
constexpr int kMaxTiles = 4096;             // per subgrid: the counts of a block in shared memory

// The subgrid whose list holds visibility i (the last s with offs[s] <= i; -1
// if its list is malformed or does not hold i), and the end of that list.
__device__ __forceinline__ int list_of(const int64_t *__restrict__ offs, int n_subgrids, int64_t n_vis, int64_t i,
                                       int64_t &end)
{
    int lo = 0, hi = n_subgrids - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (offs[mid] <= i)
            lo = mid;
        else
            hi = mid - 1;
    }
    const int64_t first = offs[lo];
    end = offs[lo + 1];
    return first >= 0 && first <= i && i < end && end <= n_vis ? lo : -1;
}

// Block b: visibilities [b kPiece, (b + 1) kPiece), list by list.  kPlace:
// write the records at the tiles' cursors; otherwise add to the tiles'
// counts, count the invalid visibilities and zero their results.
template <bool kPlace>
__global__ void __launch_bounds__(kBinThreads)
bin_kernel(const Geometry g, const Tiling t, const int64_t *__restrict__ offs, int n_subgrids, int64_t n_vis,
           const double *__restrict__ uvw, int *__restrict__ counts, BinRecord *__restrict__ records,
           float2 *__restrict__ vis_out, DeviceStatus *__restrict__ status)
{
    extern __shared__ int local[];          // [tiles] counts, then (kPlace) the places handed out
    pdl_trigger();
    pdl_wait();                             // cleared counters; kPlace: the cursors
    const int tid = threadIdx.x, tiles = t.nx * t.ny;
    const unsigned mask_x = (1u << t.lx) - 1, mask_y = (1u << t.ly) - 1;
    const int64_t piece_end = min((int64_t)(blockIdx.x + 1) * kPiece, n_vis);
    for (int64_t at = (int64_t)blockIdx.x * kPiece; at < piece_end;) {
        int64_t end;
        const int s = list_of(offs, n_subgrids, n_vis, at, end);
        if (s < 0) {                        // malformed offsets: nothing is done for this visibility
            ++at;
            continue;
        }
        const int n = (int)(min(end, piece_end) - at);
        for (int k = tid; k < tiles; k += kBinThreads)
            local[k] = 0;
        __syncthreads();
        // this thread's visibilities: tile and rank in the block's share of it
        int tile[kPerThread], rank[kPerThread];
        BinRecord rec[kPlace ? kPerThread : 1];
        int bad = 0;
#pragma unroll
        for (int j = 0; j < kPerThread; ++j) {
            const int k = tid + j * kBinThreads;
            tile[j] = -1;
            if (k < n) {
                const double *p = uvw + 3 * (at + k);
                VisCoords c;
                bool valid = visibility_coords(__ldg(p), __ldg(p + 1), __ldg(p + 2), g, c);
#ifdef DEGRID_BOUNDS_CHECK
                if (valid)
                    valid = indices_in_bounds((c.y0 * g.nx + c.x0) * g.nz + c.z0, c.fu, c.fv, c.fw, g, status);
#endif
                if (valid) {
                    tile[j] = (c.y0 >> t.ly) * t.nx + (c.x0 >> t.lx);
                    rank[j] = atomicAdd(local + tile[j], 1);
                    if (kPlace)
                        rec[j] = BinRecord{(unsigned)c.fu | ((unsigned)c.x0 & mask_x) << kBinRowBits,
                                           (unsigned)c.fv | ((unsigned)c.y0 & mask_y) << kBinRowBits, (unsigned)c.fw,
                                           (unsigned)(at + k)};
                } else if (!kPlace) {
                    ++bad;
                    if (vis_out)
                        vis_out[at + k] = make_float2(0.f, 0.f);
                }
            }
        }
        if (!kPlace) {
            bad = __reduce_add_sync(kFull, bad);
            if ((tid & 31) == 0 && bad)
                atomicAdd(&status->n_invalid, (unsigned long long)bad);
        }
        __syncthreads();
        int *global = counts + (int64_t)s * tiles;
        for (int k = tid; k < tiles; k += kBinThreads)
            if (local[k]) {
                if (kPlace)
                    local[k] = atomicAdd(global + k, local[k]);     // first place of the block's share
                else
                    atomicAdd(global + k, local[k]);
            }
        __syncthreads();
        if (kPlace) {
#pragma unroll
            for (int j = 0; j < kPerThread; ++j)
                if (tile[j] >= 0)
                    records[local[tile[j]] + rank[j]] = rec[j];
            __syncthreads();                // the places have been read
        }
        at += n;
    }
}

// Block s: the tiles' counts become the cursors their records start at, the
// items of the subgrid are appended, and its offsets are checked.  A thread
// per tile: a round over the tiles is a chain of latencies (gridding 200,000
// visibilities on 8 subgrids of 1024 tiles: 89 -> 84 us a call against 256
// threads).
__global__ void __launch_bounds__(kTilesThreads)
bin_tiles_kernel(const Tiling t, const int64_t *__restrict__ offs, int n_subgrids, int64_t n_vis,
                 int *__restrict__ counts, BinItem *__restrict__ items, int *__restrict__ n_items,
                 DeviceStatus *__restrict__ status)
{
    __shared__ int warp_vis[kTilesThreads / kWarp], warp_items[kTilesThreads / kWarp];
    __shared__ int item_base, all_vis;
    pdl_trigger();
    pdl_wait();                         // the counts
    const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int threads = blockDim.x;
    const int64_t lo = offs[s], hi = offs[s + 1];
    if (s == 0 && tid == 0 && (lo != 0 || offs[n_subgrids] != n_vis))
        atomicOr(&status->flags, kFlagOffsets);
    if (!(lo >= 0 && lo <= hi && hi <= n_vis)) {
        if (tid == 0)
            atomicOr(&status->flags, kFlagOffsets);
        return;                         // (nothing was counted)
    }
    const int tiles = t.nx * t.ny;
    int *c = counts + (long long)s * tiles;
    long long done = lo;                // records of the tiles before
    for (int base = 0; base < tiles; base += threads) {
        const int k = base + tid;
        const int n = k < tiles ? c[k] : 0;
        const int m = (n + kItemVis - 1) / kItemVis;
        int sn = n, sm = m;             // inclusive sums over the block
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int a = __shfl_up_sync(kFull, sn, d), b = __shfl_up_sync(kFull, sm, d);
            if (lane >= d) {
                sn += a;
                sm += b;
            }
        }
        if (lane == 31) {
            warp_vis[wid] = sn;
            warp_items[wid] = sm;
        }
        __syncthreads();
        if (wid == 0) {                 // sums of the warps before each; their total
            const bool in = lane < threads / kWarp;
            const int v = in ? warp_vis[lane] : 0, i = in ? warp_items[lane] : 0;
            int sv = v, si = i;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int a = __shfl_up_sync(kFull, sv, d), b = __shfl_up_sync(kFull, si, d);
                if (lane >= d) {
                    sv += a;
                    si += b;
                }
            }
            if (in) {
                warp_vis[lane] = sv - v;
                warp_items[lane] = si - i;
            }
            if (lane == 31) {
                all_vis = sv;
                item_base = si ? atomicAdd(n_items, si) : 0;
            }
        }
        __syncthreads();
        sn += warp_vis[wid];
        sm += warp_items[wid];
        if (k < tiles) {
            const long long start = done + sn - n;
            c[k] = (int)start;
            // the tile's records in m items of nearly equal size
            for (int q = 0; q < m; ++q) {
                const int a = (int)((long long)n * q / m), b = (int)((long long)n * (q + 1) / m);
                items[item_base + sm - m + q] = BinItem{s, k % t.nx, k / t.nx, b - a, start + a, 0};
            }
        }
        done += all_vis;
        __syncthreads();                // the sums have been read
    }
}

}  // namespace
}  // namespace dg

namespace {

long long tiles_of(const degrid_plan *p, dg::TileShape shape, int n_subgrids)
{
    const dg::Tiling t = dg::tiling_of(p->geo, shape);
    return (long long)t.nx * t.ny * n_subgrids;
}

// Largest buffer sizes of this many visibilities and tiles.
long long items_of(long long n_vis, long long tiles) { return n_vis / dg::kItemVis + tiles; }

}  // namespace

bool dg_bins_worth(const degrid_plan *p, dg::TileShape shape, int n_subgrids, long long n_vis)
{
    const dg::Tiling t = dg::tiling_of(p->geo, shape);
    return n_vis >= shape.min_vis + shape.min_per_tile * tiles_of(p, shape, n_subgrids) && n_vis <= (1ll << 26) &&
           (long long)t.nx * t.ny <= dg::kMaxTiles && n_subgrids <= 65535 &&
           p->geo.nx >= 48 && p->geo.ny >= 48;      // a region fits the subgrid
}

bool dg_bins_reserve(degrid_plan *p, cudaStream_t st, int n_subgrids, long long n_vis)
{
    if (!p->bins) {
        p->bins = new (std::nothrow) dg_bins();
        if (!p->bins)
            return false;
    }
    dg_bins *b = p->bins;
    // for calls in both directions: growing the workspace costs a synchronisation
    const long long td = tiles_of(p, kDegridTile, n_subgrids), tg = tiles_of(p, kGridTile, n_subgrids);
    const long long tiles = td > tg ? td : tg, items = items_of(n_vis, tiles);
    if (n_vis <= b->cap_records && tiles <= b->cap_tiles && items <= b->cap_items)
        return true;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
        return false;
    if (b->buffer) {
        cudaDeviceSynchronize();        // earlier calls may still use what is freed
        cudaFree(b->buffer);
    }
    // grown to the largest of each
    const long long nr = n_vis > b->cap_records ? n_vis : b->cap_records;
    const long long ni = items > b->cap_items ? items : b->cap_items;
    const long long nt = tiles > b->cap_tiles ? tiles : b->cap_tiles;
    *b = dg_bins();
    const size_t bytes = sizeof(dg::BinRecord) * (size_t)nr + sizeof(dg::BinItem) * (size_t)ni +
                         sizeof(int) * (size_t)(nt + 2);
    if (cudaMalloc(&b->buffer, bytes) != cudaSuccess) {
        cudaGetLastError();
        b->buffer = nullptr;
        return false;
    }
    b->records = static_cast<dg::BinRecord *>(b->buffer);
    b->items = reinterpret_cast<dg::BinItem *>(b->records + nr);
    b->counters = reinterpret_cast<int *>(b->items + ni);
    b->cap_records = nr;
    b->cap_items = ni;
    b->cap_tiles = nt;
    return true;
}

cudaError_t dg_bins_sort(degrid_plan *p, cudaStream_t st, dg::TileShape shape, int n_subgrids,
                         long long n_vis, const double *uvw, const int64_t *vis_offsets, float *vis_out,
                         dg::Bins *out)
{
    using namespace dg;
    dg_bins *b = p->bins;
    const Tiling t = tiling_of(p->geo, shape);
    cudaError_t e = cudaMemsetAsync(b->counters, 0, sizeof(int) * (size_t)(tiles_of(p, shape, n_subgrids) + 2), st);
    if (e != cudaSuccess)
        return e;
    int *counts = b->counters + 2;
    const dim3 blocks((unsigned)((n_vis + kPiece - 1) / kPiece));
    const size_t smem = sizeof(int) * (size_t)t.nx * t.ny;      // at most 16 KB
    const int rounded = (t.nx * t.ny + kWarp - 1) / kWarp * kWarp;
    const int tile_threads = rounded < kTilesThreads ? rounded : kTilesThreads;
    float2 *zeros = reinterpret_cast<float2 *>(vis_out);
    bin_kernel<false><<<blocks, kBinThreads, smem, st>>>(p->geo, t, vis_offsets, n_subgrids, (int64_t)n_vis, uvw, counts,
                                                         b->records, zeros, p->status);
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = launch_pdl(bin_tiles_kernel, dim3((unsigned)n_subgrids), dim3((unsigned)tile_threads), 0, st, t, vis_offsets,
                       n_subgrids, (int64_t)n_vis, counts, b->items, b->counters, p->status);
    if (e == cudaSuccess)
        e = launch_pdl(bin_kernel<true>, blocks, dim3(kBinThreads), smem, st, p->geo, t, vis_offsets, n_subgrids,
                       (int64_t)n_vis, uvw, counts, b->records, zeros, p->status);
    *out = Bins{t, b->records, b->items, b->counters, b->counters + 1};
    return e;
}

void dg_bins_free(degrid_plan *p)
{
    if (!p->bins)
        return;
    cudaFree(p->bins->buffer);
    delete p->bins;
    p->bins = nullptr;
}
