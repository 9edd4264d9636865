// Degridding with a non-separable 2D G_uv table: every visibility has its own
// 8 x 8 block of weights G[fv][fu][b][a],
//     V = sum_b sum_a G[fv][fu][b][a] M[b][a],   M[b][a] = sum_c g_w[c] s[y0+b][x0+a][z0+c].
//
// A persistent grid of warps walks chunks in steps of 32 visibilities; lane i
// owns visibility i of the step from the coordinates to the store.  Per step
// a warp
//  1. snaps the coordinates of the next step (loaded a step before) while the
//     weight blocks of the current one are on their way;
//  2. loads the coordinates of the step after that;
//  3. builds the footprints M it does not hold yet, sums and stores;
//  4. starts the copies (cp.async) of the next step's blocks, 256 bytes per
//     visibility, half a warp per block.
//
// M depends only on the footprint start and the w row, which consecutive
// visibilities of a dense list share: the warp keeps the last kSlots of them
// in shared memory and every lane reads the one of its own visibility.  Lanes
// of one run read the same address (a broadcast).  Slots start 16 bytes
// further into the 128-byte bank line than the slot before, so a step that
// holds up to kSlots runs is built, with the loads of its footprints in
// flight together, and summed once.
//
// What bounds it is the L1 data path, a line or 128 bytes of shared memory
// per cycle: a visibility's weights take two lines in and two reads out, its
// share of M one to four reads.  When four lanes shared a visibility and read
// the table themselves its weights took eight line accesses, and a step with
// several runs one pass per run and eight visibilities: 166 us against 88 for
// 2.5M visibilities on 24 subgrids' lines and arcs (123 with the weights loaded
// by every lane itself, a line access per 32 bytes), 298 against 289 for 16M on
// 64 subgrids' lines (336 when every visibility's block was copied: its 4.1 GB
// come from L2).
#include "footprint.cuh"
#include "pipeline.cuh"

namespace dg {
namespace {

constexpr int kMaxWarps = 8;                // per CTA
constexpr int kSlots = 8;                   // footprints a warp holds (a power of two)
constexpr int kBlock = kUV * kUV;           // weights of a visibility
constexpr int kPieces = kBlock / 4;         // 16-byte pieces of them

// M[b][a] of one footprint; the padding moves the next slot by one 16-byte
// bank group.
struct alignas(16) MSlot {
    float2 m[kUV][kUV];
    float2 pad[2];
};

struct alignas(128) WarpSmem {
    float4 w[kBatch][kPieces];              // weight blocks of the step (piece q of row r at place(r, q))
    MSlot slot[kSlots];
    int blk[kBatch];                        // which block each row of w holds
};

// Place of piece q of row r in the stage: the same piece of eight consecutive
// rows lies in eight different bank groups.
__device__ __forceinline__ int place(int r, int q) { return q ^ (r & 7); }

// What the M builds of a warp need besides the footprint.
struct BuildArgs {
    const void *subgrids;
    const float4 *wtab;             // w table in shared memory, or nullptr
    const float *gwt;               // w table in global memory
    bool vec_ok;
    int lane;
};

// This lane's two points of M for footprint `key`, w row fw of the subgrid at
// element `base`: column lane & 7 of rows lane >> 3 and (lane >> 3) + 4.
template <int DT>
__device__ __forceinline__ void build_points(float2 (&m)[2], int64_t base, int key, int fw, const Geometry &g,
                                             const BuildArgs &A)
{
    const float4 gw = A.wtab ? A.wtab[fw] : __ldg(reinterpret_cast<const float4 *>(A.gwt) + fw);
    const int64_t col = base + key + (int64_t)(A.lane & 7) * g.nz + (int64_t)(A.lane >> 3) * g.row_stride;
    const bool vec = vec_footprint<DT>(A.vec_ok, key);
#pragma unroll
    for (int k = 0; k < 2; ++k)
        m[k] = footprint_point<DT>(A.subgrids, col + (int64_t)(4 * k) * g.row_stride, gw, vec);
}

__device__ __forceinline__ void store_points(MSlot &slot, const float2 (&m)[2], int lane)
{
    (&slot.m[0][0])[lane] = m[0];
    (&slot.m[4][0])[lane] = m[1];
}

// A lane's visibility.
struct Vis {
    int key;            // footprint start, -1: invalid or past the end of the step
    int fw;             // w row
    int blk;            // weight block fv * O + fu
    int row;            // row of the stage that holds it
};

__device__ __forceinline__ Vis snap_step(const Batch &b, const Coords3 &c, const Geometry &g, DeviceStatus *status,
                                         int lane)
{
    const bool in = lane < b.n;
    VisCoords vc;
    bool valid = in && visibility_coords(c.u, c.v, c.w, g, vc);
#ifdef DEGRID_BOUNDS_CHECK
    if (valid)
        valid = indices_in_bounds((vc.y0 * g.nx + vc.x0) * g.nz + vc.z0, vc.fu, vc.fv, vc.fw, g, status);
#endif
    const unsigned bad = __ballot_sync(kFull, in && !valid);
    if (lane == 0 && bad)
        atomicAdd(&status->n_invalid, (unsigned long long)__popc(bad));
    Vis r;
    r.key = valid ? (vc.y0 * g.nx + vc.x0) * g.nz + vc.z0 : -1;
    r.fw = valid ? vc.fw : 0;
    r.blk = valid ? (vc.fv << g.log2_uv_os) + vc.fu : 0;
    r.row = lane;
    return r;
}

// Starts the copies of a step's weight blocks (one cp.async group).
// Consecutive visibilities with one block share a row of the stage: on dense
// lists the snapped offsets move slower than the visibilities.
__device__ __forceinline__ void copy_weights(WarpSmem &ws, Vis &v, const float *__restrict__ g2, int lane)
{
    const int before = __shfl_up_sync(kFull, v.blk, 1);
    const bool head = lane == 0 || v.blk != before;
    const unsigned heads = __ballot_sync(kFull, head);
    const int rows = __popc(heads), q = lane & (kPieces - 1);
    if (rows > kBatch / 2) {
        v.row = lane;
#pragma unroll
        for (int i = 0; i < kBatch; i += 2) {
            const int r = i + (lane >> 4);
            const int blk = __shfl_sync(kFull, v.blk, r);
            cp_async16(smem_u32(&ws.w[r][place(r, q)]), g2 + (size_t)blk * kBlock + 4 * q);
        }
    } else {
        v.row = __popc(heads & (kFull >> (31 - lane))) - 1;
        if (head)
            ws.blk[v.row] = v.blk;
        __syncwarp();
        for (int i = 0; i < rows; i += 2) {
            const int r = i + (lane >> 4);
            if (r < rows)
                cp_async16(smem_u32(&ws.w[r][place(r, q)]), g2 + (size_t)ws.blk[r] * kBlock + 4 * q);
        }
    }
    cp_async_commit();
}

// (Q0 + Q2) + (Q1 + Q3), the order every kernel of the library uses; the
// compensated form makes the three additions error-free, sums their errors
// and adds them back once.
template <bool COMP>
__device__ __forceinline__ float combine(const float (&q)[4])
{
    if (!COMP)
        return (q[0] + q[2]) + (q[1] + q[3]);
    float e0, e1, e;
    const float s0 = two_sum(q[0], q[2], e0), s1 = two_sum(q[1], q[3], e1);
    const float v = two_sum(s0, s1, e);
    return v + (e + (e0 + e1));
}

// Sum of row b of the footprint with row b of the weights in stage row `row`,
// an FMA chain of (re, im) pairs.
__device__ __forceinline__ float2 row_sum(const float4 (&m)[4], const WarpSmem &ws, int row, int b)
{
    const float4 w0 = ws.w[row][place(row, 2 * b)], w1 = ws.w[row][place(row, 2 * b + 1)];
    float2 t = __fmul2_rn(make_float2(m[0].x, m[0].y), make_float2(w0.x, w0.x));
    t = __ffma2_rn(make_float2(m[0].z, m[0].w), make_float2(w0.y, w0.y), t);
    t = __ffma2_rn(make_float2(m[1].x, m[1].y), make_float2(w0.z, w0.z), t);
    t = __ffma2_rn(make_float2(m[1].z, m[1].w), make_float2(w0.w, w0.w), t);
    t = __ffma2_rn(make_float2(m[2].x, m[2].y), make_float2(w1.x, w1.x), t);
    t = __ffma2_rn(make_float2(m[2].z, m[2].w), make_float2(w1.y, w1.y), t);
    t = __ffma2_rn(make_float2(m[3].x, m[3].y), make_float2(w1.z, w1.z), t);
    return __ffma2_rn(make_float2(m[3].z, m[3].w), make_float2(w1.w, w1.w), t);
}

__device__ __forceinline__ void load_row(float4 (&m)[4], const MSlot &slot, int b)
{
    const float4 *p = reinterpret_cast<const float4 *>(&slot.m[b][0]);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        m[k] = p[k];
}

// The lane's visibility from the footprint in `slot`: quarter j is the sum of
// rows 2j and 2j + 1.
template <bool COMP>
__device__ __forceinline__ float2 sum_lane(const MSlot &slot, const WarpSmem &ws, int row)
{
    float qx[4], qy[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float2 R[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float4 m[4];
            load_row(m, slot, 2 * j + i);
            R[i] = row_sum(m, ws, row, 2 * j + i);
        }
        const float2 q = __fadd2_rn(R[0], R[1]);
        qx[j] = q.x;
        qy[j] = q.y;
    }
    return make_float2(combine<COMP>(qx), combine<COMP>(qy));
}

// The same when the whole step is on one footprint: lanes l and l + 16 take
// four rows each for both of their visibilities, which halves the reads of the
// footprint, and exchange two quarters.  (Neighbouring lanes, so that both
// rows are read within eight lanes, gained nothing: 318 us for 16M
// visibilities on 64 subgrids' lines, 314 without sharing, 289 like this.)
template <bool COMP>
__device__ __forceinline__ float2 sum_pair(const MSlot &slot, const WarpSmem &ws, int row, int lane)
{
    const int h = lane >> 4, other = __shfl_xor_sync(kFull, row, 16);
    const int ra = h ? other : row, rb = h ? row : other;       // stage rows of the lower and the upper lane
    float2 qa[2], qb[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float2 A[2], B[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int b = 4 * h + 2 * j + i;
            float4 m[4];
            load_row(m, slot, b);
            A[i] = row_sum(m, ws, ra, b);
            B[i] = row_sum(m, ws, rb, b);
        }
        qa[j] = __fadd2_rn(A[0], A[1]);
        qb[j] = __fadd2_rn(B[0], B[1]);
    }
    float qx[4], qy[4];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float2 give = h ? qa[j] : qb[j], keep = h ? qb[j] : qa[j];
        const float2 got = make_float2(__shfl_xor_sync(kFull, give.x, 16), __shfl_xor_sync(kFull, give.y, 16));
        qx[j] = h ? got.x : keep.x;
        qy[j] = h ? got.y : keep.y;
        qx[j + 2] = h ? keep.x : got.x;
        qy[j + 2] = h ? keep.y : got.y;
    }
    return make_float2(combine<COMP>(qx), combine<COMP>(qy));
}

// The most recently built footprint of a warp: (key, fw) of the current
// subgrid is in slot `slot` (key -2: none).
struct MCache {
    int key, fw, slot;
};

// A step that does not continue the cached run alone: its runs (maximal
// sequences of equal footprint and w row) are built up to kSlots at a time,
// two footprints' loads in flight together, and each round is summed once,
// every lane from the slot of its own run.
template <int DT, bool COMP>
__device__ __forceinline__ float2 sum_runs(MCache &mc, WarpSmem &ws, int64_t base, const Vis &v, const Geometry &g,
                                           const BuildArgs &A)
{
    const int lane = A.lane;
    const int kp = __shfl_up_sync(kFull, v.key, 1), fp = __shfl_up_sync(kFull, v.fw, 1);
    unsigned heads = __ballot_sync(kFull, v.key >= 0 && (lane == 0 || v.key != kp || v.fw != fp));
    const int run = __popc(heads & (0xffffffffu >> (31 - lane))) - 1;
    const int n_runs = __popc(heads);
    float2 V = make_float2(0.f, 0.f);
    for (int first = 0; first < n_runs; first += kSlots) {
        const int n = min(kSlots, n_runs - first);
        __syncwarp();                   // the slots have been read
        int todo = n;
        {   // a first run that continues the cached one needs no build
            const int src = __ffs(heads) - 1;
            const int key = __shfl_sync(kFull, v.key, src), fw = __shfl_sync(kFull, v.fw, src);
            if (key == mc.key && fw == mc.fw) {
                heads &= heads - 1;
                --todo;
            }
        }
        const int start = (mc.slot + (todo == n ? 1 : 0)) & (kSlots - 1);   // slot of the round's first run
        while (todo > 0) {
            const int src0 = __ffs(heads) - 1;
            heads &= heads - 1;
            const bool two = todo > 1;
            const int src1 = two ? __ffs(heads) - 1 : src0;
            if (two)
                heads &= heads - 1;
            const int k0 = __shfl_sync(kFull, v.key, src0), f0 = __shfl_sync(kFull, v.fw, src0);
            const int k1 = __shfl_sync(kFull, v.key, src1), f1 = __shfl_sync(kFull, v.fw, src1);
            float2 m0[2], m1[2];
            build_points<DT>(m0, base, k0, f0, g, A);
            build_points<DT>(m1, base, k1, f1, g, A);
            mc.slot = (mc.slot + 1) & (kSlots - 1);
            store_points(ws.slot[mc.slot], m0, lane);
            if (two) {
                mc.slot = (mc.slot + 1) & (kSlots - 1);
                store_points(ws.slot[mc.slot], m1, lane);
            }
            mc.key = k1;
            mc.fw = f1;
            todo -= two ? 2 : 1;
        }
        __syncwarp();
        const bool mine = v.key >= 0 && run >= first && run < first + n;
        const float2 x = sum_lane<COMP>(ws.slot[(start + (mine ? run - first : 0)) & (kSlots - 1)], ws, v.row);
        if (mine)
            V = x;
    }
    return V;
}

template <int DT, bool COMP>
__global__ void __launch_bounds__(kMaxWarps * kWarp, 2)
degrid_2d_kernel(const Geometry g, const void *__restrict__ subgrids, const float *__restrict__ scale,
                 const double *__restrict__ uvw, const float *__restrict__ gwt, const Schedule sched,
                 float2 *__restrict__ vis_out, DeviceStatus *__restrict__ status, const bool vec_ok,
                 const float *__restrict__ g2, const bool prefetch_uvw)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // [w table (optional)] [one WarpSmem per warp]
    WarpSmem &ws = reinterpret_cast<WarpSmem *>(smem_raw + wtable_bytes(g))[threadIdx.x >> 5];
    const float4 *wtab = load_wtable(g, gwt, smem_raw);
    const int lane = threadIdx.x & 31;
    const BuildArgs A{subgrids, wtab, gwt, vec_ok, lane};

    pdl_wait();                         // the chunk table is complete
    Claimer claimer(sched, lane, Prefetch{prefetch_uvw ? uvw : nullptr, 3 * (int)sizeof(double), nullptr, 0});
    Batch bA = claimer.claim();         // the step being summed
    if (bA.n == 0)
        return;
    Vis vA = snap_step(bA, load_uvw(uvw, bA, lane), g, status, lane);
    copy_weights(ws, vA, g2, lane);
    Batch bB = claimer.advance(bA);     // the step after it, its coordinates in registers
    Coords3 c = load_uvw(uvw, bB, lane);

    MCache mc{-2, -1, 0};
    int m_s = -1;
    int64_t base = 0;
    float sc = 1.f;
    while (true) {
        Vis vB = snap_step(bB, c, g, status, lane);
        const Batch bC = claimer.advance(bB);
        c = load_uvw(uvw, bC, lane);

        if (bA.s != m_s) {
            m_s = bA.s;
            mc.key = -2;
            base = (int64_t)bA.s * g.plane;
            if (DT != DG_C64)
                sc = __ldg(scale + bA.s);
        }
        cp_async_wait<0>();
        __syncwarp();                   // every lane's copies of the weights
        float2 V;
        if (__all_sync(kFull, vA.key == mc.key && vA.fw == mc.fw))
            V = sum_pair<COMP>(ws.slot[mc.slot], ws, vA.row, lane);   // the step continues the cached run
        else
            V = sum_runs<DT, COMP>(mc, ws, base, vA, g, A);
        if (DT != DG_C64)
            V = __fmul2_rn(V, make_float2(sc, sc));
        if (lane < bA.n)
            vis_out[bA.b0 + lane] = V;
        if (bB.n == 0)
            break;
        __syncwarp();                   // the weights have been read
        copy_weights(ws, vB, g2, lane);
        vA = vB;
        bA = bB;
        bB = bC;
    }
}

size_t smem_bytes(const degrid_plan *p)
{
    return wtable_bytes_host(p->geo) + sizeof(WarpSmem) * (size_t)p->warps_per_block;
}

// Dynamic shared memory opened so far for a kernel instance on a device.
template <int DT, bool COMP>
std::atomic<size_t> &smem_record(int device)
{
    static std::atomic<size_t> table[kMaxDevices];
    return dg_smem_record(table, device);
}

template <int DT, bool COMP>
cudaError_t launch(degrid_plan *p, cudaStream_t st, const void *subgrids, const float *scale, const double *uvw,
                   float2 *out, const Schedule &sched, int grid_blocks)
{
    const size_t smem = smem_bytes(p);
    const cudaError_t e = dg_open_smem(smem_record<DT, COMP>(p->device), degrid_2d_kernel<DT, COMP>, smem);
    if (e != cudaSuccess)
        return e;
    // 16-byte footprint loads need an aligned stack and nz a multiple of the
    // elements per 16 bytes
    const bool vec_ok = (reinterpret_cast<uintptr_t>(subgrids) & 15) == 0 &&
                        p->geo.nz % Storage<DT>::kQuad == 0;
    return launch_pdl(degrid_2d_kernel<DT, COMP>, dim3(grid_blocks), dim3(p->warps_per_block * kWarp), smem, st,
                      p->geo, subgrids, scale, uvw, (const float *)p->gw, sched, out, p->status, vec_ok,
                      (const float *)p->guv2, !p->host_inputs);
}

template <int DT, bool COMP>
int max_blocks(degrid_plan *p)
{
    int n = 0;
    const size_t smem = smem_bytes(p);
    if (dg_open_smem(smem_record<DT, COMP>(p->device), degrid_2d_kernel<DT, COMP>, smem) != cudaSuccess)
        return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, degrid_2d_kernel<DT, COMP>, p->warps_per_block * kWarp,
                                                      smem) != cudaSuccess)
        return 1;
    return n > 0 ? n : 1;
}

}  // namespace
}  // namespace dg

cudaError_t dg_launch_degrid_2d(degrid_plan *p, cudaStream_t st, const void *subgrids, const float *scale,
                                const double *uvw, float *out_f, int grid_blocks)
{
    using namespace dg;
    Schedule sched{p->chunks, p->n_chunks, p->work_counter};
    float2 *out = reinterpret_cast<float2 *>(out_f);
    const auto run = [&](auto plain, auto comp) { return (p->compensated ? comp : plain)(p, st, subgrids, scale, uvw, out, sched, grid_blocks); };
    switch (p->dtype) {
    case DG_C64: return run(launch<DG_C64, false>, launch<DG_C64, true>);
    case DG_C32_F16: return run(launch<DG_C32_F16, false>, launch<DG_C32_F16, true>);
    case DG_C32_BF16: return run(launch<DG_C32_BF16, false>, launch<DG_C32_BF16, true>);
    }
    return cudaErrorInvalidValue;
}

int dg_max_blocks_per_sm_degrid_2d(degrid_plan *p)
{
    using namespace dg;
    switch (p->dtype) {
    case DG_C64: return p->compensated ? max_blocks<DG_C64, true>(p) : max_blocks<DG_C64, false>(p);
    case DG_C32_F16: return p->compensated ? max_blocks<DG_C32_F16, true>(p) : max_blocks<DG_C32_F16, false>(p);
    case DG_C32_BF16: return p->compensated ? max_blocks<DG_C32_BF16, true>(p) : max_blocks<DG_C32_BF16, false>(p);
    }
    return 1;
}
