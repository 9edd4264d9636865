// Degridding kernel (paper Section "Implementation": kernel D1 and its
// variants), re-designed for sm_103a.
//
// Work decomposition (pipeline.cuh).  A persistent grid of warps walks chunks
// of consecutive visibilities of one subgrid in steps of 64: lane i owns
// visibilities i and i + 32 of the step from the coordinates to the store.
// Per step a warp
//  1. snaps the coordinates of the next step (loaded one step before; the
//     next chunk's are prefetched into L2 when its descriptor arrives), while
//     the table rows of the current step are on their way;
//  2. loads the coordinates of the step after that;
//  3. builds the footprints M it does not hold yet, sums and stores;
//  4. starts the copies (cp.async) of the next step's g_u and g_v rows into
//     the warp's shared-memory stage, two lanes per 32-byte row.
//
// Footprint sum.  The separable weights let the 8 x 8 x 4 sum be taken in
// three contractions,
//     V = sum_b g_v[b] sum_a g_u[a] M[b][a],   M[b][a] = sum_c g_w[c] s[y0+b][x0+a][z0+c],
// and M depends only on the footprint start and the w-kernel row.  On a dense
// list hundreds of consecutive visibilities share both (the reuse the paper
// notes for D1), so M is computed once per run, by the whole warp, into one
// of the warp's shared-memory slots, and each visibility then costs 72
// complex x real products instead of 256.  Every lane reads M from shared
// memory: lanes of one run read the same address (a broadcast), and when both
// visibilities of every lane share a run, one read serves two products.
// Slots start 16 bytes further into the 128-byte bank line than the slot
// before, so lanes of several runs read different banks: a step that holds up
// to kSlots runs is built and summed in one pass.
//
// Every operation and its order are those of the gather, tile and 2D-table
// kernels, so all agree bit for bit.
//
// What bounds it.  16M visibilities on 64 subgrids' lines take 211 us, 260
// cycles per SM and 64 visibilities.  Of those the requests to L1 and L2 take
// about 175 (128 table rows at 1.06 cycles each, measured in isolation,
// whatever the copy; the coordinates and the output), the load/store data
// path 165, the six FP64-to-int32 conversions of the snap 96 (16 cycles per
// warp instruction), the packed FMAs 76; 16 warps per SM overlap them at 62%.
// Measured and slower: the rows loaded into registers by each lane (249 us:
// a data-path cycle per row), two row stages (278: the copies queue up before
// the coordinate loads), coordinates copied to shared memory (225), 24 warps
// with 80 registers (242).
//
// Four lanes per visibility, each with two rows of M in registers, took 222
// us here and summed a step with several runs once per run and eight
// visibilities: 14M visibilities on 96 subgrids' lines and arcs of uneven
// length took 284 us, and take 237.
#include <type_traits>

#include "footprint.cuh"
#include "pipeline.cuh"

namespace dg {
namespace {

constexpr int kMaxWarps = 8;                // per CTA
constexpr int kStepVis = 2 * kBatch;        // visibilities per pipeline step: two per lane
constexpr int kSlots = 8;                   // footprints a warp holds (a power of two)

// M[b][a] of one footprint; the padding moves the next slot by one 16-byte
// bank group.
struct alignas(16) MSlot {
    float2 m[kUV][kUV];
    float2 pad[2];
};

struct alignas(128) WarpSmem {
    RowStage st[2];             // [half]
    MSlot slot[kSlots];
};

// A step: subgrid, visibilities left in its chunk from here on (0: no work
// left), and where this lane's first visibility is read and written.
struct Step {
    int s, n;
    const double *uvw;
    float2 *out;
};

// Steps of the chunks (or pieces) a warp claims.
template <class Claim>
struct Steps {
    Claim claimer;
    const double *uvw;          // this lane's offset included
    float2 *out;

    __device__ Step claim()
    {
        const Batch b = claimer.claim();
        return Step{b.s, (int)(b.end - b.b0), uvw + 3 * b.b0, out + b.b0};
    }

    __device__ Step advance(const Step &p)
    {
        if (p.n == 0)
            return p;
        if (p.n <= kStepVis)
            return claim();
        return Step{p.s, p.n - kStepVis, p.uvw + 3 * kStepVis, p.out + kStepVis};
    }
};

// Coordinates of the lane's two visibilities (zeros past the end).
__device__ __forceinline__ void load_coords(Coords3 (&c)[2], const Step &p, int lane)
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        c[h] = Coords3{0.0, 0.0, 0.0};
        if (lane + kBatch * h < p.n) {
            c[h].u = __ldg(p.uvw + 3 * kBatch * h);
            c[h].v = __ldg(p.uvw + 3 * kBatch * h + 1);
            c[h].w = __ldg(p.uvw + 3 * kBatch * h + 2);
        }
    }
}

// ---- the factored sum -------------------------------------------------------

// What the M builds of a warp need besides the footprint.
struct BuildArgs {
    const void *subgrids;
    const float4 *wtab;             // w table in shared memory, or nullptr
    const float *gwt;               // w table in global memory
    bool vec_ok;
    int lane;
};

__device__ __forceinline__ float4 w_row(const BuildArgs &A, int fw)
{
    return A.wtab ? A.wtab[fw] : __ldg(reinterpret_cast<const float4 *>(A.gwt) + fw);
}

// This lane's two points of M for footprint `key`, w row fw of the subgrid at
// element `base`: column lane & 7 of rows lane >> 3 and (lane >> 3) + 4.
template <int DT>
__device__ __forceinline__ void build_points(float2 (&m)[2], int64_t base, int key, int fw, const Geometry &g,
                                             const BuildArgs &A)
{
    const float4 gw = w_row(A, fw);
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

// The two visibilities of a lane in a step.
struct Vis2 {
    int key[2];         // footprint start, -1: invalid or past the end of the step
    int fw[2];          // w row
    int ru[2], rv[2];   // g_u and g_v rows (-1 with key -1)
};

__device__ __forceinline__ Vis2 snap_step(const Step &b, const Coords3 (&c)[2], const Geometry &g,
                                          DeviceStatus *status, int lane)
{
    Vis2 r;
    bool bad[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const bool in = lane + kBatch * h < b.n;
        VisCoords vc;
        bool valid = in && visibility_coords(c[h].u, c[h].v, c[h].w, g, vc);
#ifdef DEGRID_BOUNDS_CHECK
        if (valid)
            valid = indices_in_bounds((vc.y0 * g.nx + vc.x0) * g.nz + vc.z0, vc.fu, vc.fv, vc.fw, g, status);
#endif
        r.key[h] = valid ? (vc.y0 * g.nx + vc.x0) * g.nz + vc.z0 : -1;
        r.fw[h] = valid ? vc.fw : 0;
        r.ru[h] = valid ? vc.fu : -1;
        r.rv[h] = valid ? vc.fv : -1;
        bad[h] = in && !valid;
    }
    if (__any_sync(kFull, bad[0] || bad[1])) {
        const int n = __popc(__ballot_sync(kFull, bad[0])) + __popc(__ballot_sync(kFull, bad[1]));
        if (lane == 0)
            atomicAdd(&status->n_invalid, (unsigned long long)n);
    }
    return r;
}

// A table row in registers.
struct Row8 {
    float w[kUV];
};

// Starts the copies of the step's g_u and g_v rows (two lanes per 32-byte
// row, so each row is one request; one cp.async group).  Lanes without a
// valid visibility copy nothing and drop what they sum from the stale stage:
// one row for all of them made the partial steps of small calls queue up at
// one sector of L2 (20,000 visibilities in steps of 16: 28 us against 5).
__device__ __forceinline__ void copy_rows(RowStage (&st)[2], const Vis2 &s, const float *__restrict__ guv, int lane)
{
    const int half = lane & 1;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int row = (lane >> 1) + 16 * m;
            const int xu = __shfl_sync(kFull, s.ru[h], row);
            const int xv = __shfl_sync(kFull, s.rv[h], row);
            if (xu < 0)
                continue;
            cp_async16(smem_u32(&st[h].u[row][RowStage::slot(row, half)]), guv + (size_t)xu * kUVRow + 4 * half);
            cp_async16(smem_u32(&st[h].v[row][RowStage::slot(row, half)]), guv + (size_t)xv * kUVRow + 4 * half);
        }
    cp_async_commit();
}

__device__ __forceinline__ Row8 stage_row(const float4 (&row)[2], int lane)
{
    const float4 a = row[RowStage::slot(lane, 0)], b = row[RowStage::slot(lane, 1)];
    return Row8{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}

// sum_a g[a] m[a] over one row of M (4 float4 in shared memory), as packed
// pairs (re, im) * (g, g): one FFMA2 per product, each half rounded exactly
// as a scalar FMA.
__device__ __forceinline__ float2 row_sum(const float4 (&m)[4], const Row8 &g)
{
    float2 t = __fmul2_rn(make_float2(m[0].x, m[0].y), make_float2(g.w[0], g.w[0]));
    t = __ffma2_rn(make_float2(m[0].z, m[0].w), make_float2(g.w[1], g.w[1]), t);
#pragma unroll
    for (int a = 1; a < 4; ++a) {
        t = __ffma2_rn(make_float2(m[a].x, m[a].y), make_float2(g.w[2 * a], g.w[2 * a]), t);
        t = __ffma2_rn(make_float2(m[a].z, m[a].w), make_float2(g.w[2 * a + 1], g.w[2 * a + 1]), t);
    }
    return t;
}

__device__ __forceinline__ void read_row(float4 (&m)[4], const MSlot &slot, int b)
{
    const float4 *p = reinterpret_cast<const float4 *>(&slot.m[b][0]);
#pragma unroll
    for (int a = 0; a < 4; ++a)
        m[a] = p[a];
}

// (Q0 + Q2) + (Q1 + Q3), the order every kernel of the library uses; the
// compensated form makes the three additions error-free, sums their errors
// and adds them back once.
template <bool COMP>
__device__ __forceinline__ float combine(float q0, float q1, float q2, float q3)
{
    if (!COMP)
        return (q0 + q2) + (q1 + q3);
    float e0, e1, e;
    const float s0 = two_sum(q0, q2, e0), s1 = two_sum(q1, q3, e1);
    const float v = two_sum(s0, s1, e);
    return v + (e + (e0 + e1));
}

// The lane's two visibilities from the footprints in s0 and s1 (with SHARED
// the same slot for both: read once) and their rows in the stage.  Quarter j
// is rows 2j and 2j + 1, g_v[2j + 1] R_{2j + 1} + g_v[2j] R_{2j} with
// R_b = sum_a g_u[a] M[b][a].
template <bool COMP, bool SHARED>
__device__ __forceinline__ void sum_step(float2 (&V)[2], const MSlot &s0, const MSlot &s1, const RowStage (&st)[2],
                                         int lane)
{
    float2 Q[2][4];
    const Row8 gu[2] = {stage_row(st[0].u[lane], lane), stage_row(st[1].u[lane], lane)};
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
        const float4 gv[2] = {st[0].v[lane][RowStage::slot(lane, jj)], st[1].v[lane][RowStage::slot(lane, jj)]};
#pragma unroll
        for (int j2 = 0; j2 < 2; ++j2) {
            const int j = 2 * jj + j2;
            float2 R[2][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int b = 2 * j + i;
                float4 m[4];
                read_row(m, s0, b);
                R[0][i] = row_sum(m, gu[0]);
                if (!SHARED)
                    read_row(m, s1, b);
                R[1][i] = row_sum(m, gu[1]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float ve = j2 ? gv[h].z : gv[h].x, vo = j2 ? gv[h].w : gv[h].y;
                Q[h][j] = __ffma2_rn(R[h][1], make_float2(vo, vo), __fmul2_rn(R[h][0], make_float2(ve, ve)));
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        V[h].x = combine<COMP>(Q[h][0].x, Q[h][1].x, Q[h][2].x, Q[h][3].x);
        V[h].y = combine<COMP>(Q[h][0].y, Q[h][1].y, Q[h][2].y, Q[h][3].y);
    }
}

// The most recently built footprint of a warp: (key, fw) of the current
// subgrid is in slot `slot` (key -2: none).
struct MCache {
    int key, fw, slot;
};

// A step that does not continue the cached run alone: its runs (maximal
// sequences of equal footprint and w row in list order) are built up to
// kSlots at a time, two footprints' loads in flight together, and each round
// is summed once, every lane reading the slots of its own visibilities' runs.
template <int DT, bool COMP>
__device__ __forceinline__ void sum_runs(float2 (&V)[2], MCache &mc, WarpSmem &ws, const RowStage (&st)[2],
                                         int64_t base, const Vis2 &vis,
                                         const Geometry &g, const BuildArgs &A)
{
    const int lane = A.lane;
    __syncwarp();                       // earlier steps' reads of the slots are done
    unsigned heads[2];
    int run[2];                         // run of the lane's visibilities
    {
        int kp = __shfl_up_sync(kFull, vis.key[0], 1), fp = __shfl_up_sync(kFull, vis.fw[0], 1);
        heads[0] = __ballot_sync(kFull, vis.key[0] >= 0 && (lane == 0 || vis.key[0] != kp || vis.fw[0] != fp));
        // visibility 32 follows visibility 31
        kp = __shfl_sync(kFull, lane == 31 ? vis.key[0] : vis.key[1], (lane + 31) & 31);
        fp = __shfl_sync(kFull, lane == 31 ? vis.fw[0] : vis.fw[1], (lane + 31) & 31);
        heads[1] = __ballot_sync(kFull, vis.key[1] >= 0 && (vis.key[1] != kp || vis.fw[1] != fp));
        const unsigned upto = 0xffffffffu >> (31 - lane);
        run[0] = __popc(heads[0] & upto) - 1;
        run[1] = __popc(heads[0]) + __popc(heads[1] & upto) - 1;
    }
    const int n_runs = __popc(heads[0]) + __popc(heads[1]);
    V[0] = V[1] = make_float2(0.f, 0.f);
    for (int first = 0; first < n_runs; first += kSlots) {
        const int n = min(kSlots, n_runs - first);
        int todo = n;
        const auto head = [&](int &key, int &fw) {          // takes the next run's head off the list
            const int h = heads[0] ? 0 : 1;
            const int src = __ffs(h ? heads[1] : heads[0]) - 1;
            key = __shfl_sync(kFull, h ? vis.key[1] : vis.key[0], src);
            fw = __shfl_sync(kFull, h ? vis.fw[1] : vis.fw[0], src);
            if (h)
                heads[1] &= heads[1] - 1;
            else
                heads[0] &= heads[0] - 1;
        };
        int key, fw;
        head(key, fw);
        bool have = true;               // (key, fw) is a run that is not built yet
        if (key == mc.key && fw == mc.fw) {
            --todo;                     // the first run continues the cached one
            have = false;
        }
        const int start = (mc.slot + (have ? 1 : 0)) & (kSlots - 1);
        // builds the next N runs, their loads in flight together
        const auto build = [&](auto n_runs_built) {
            constexpr int N = decltype(n_runs_built)::value;
            int k[N], f[N];
            float2 m[N][2];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                if (!have)
                    head(key, fw);
                have = false;
                k[i] = key;
                f[i] = fw;
            }
#pragma unroll
            for (int i = 0; i < N; ++i)
                build_points<DT>(m[i], base, k[i], f[i], g, A);
#pragma unroll
            for (int i = 0; i < N; ++i) {
                mc.slot = (mc.slot + 1) & (kSlots - 1);
                store_points(ws.slot[mc.slot], m[i], lane);
            }
            mc.key = key;
            mc.fw = fw;
            todo -= N;
        };
        while (todo >= 2)               // (four at a time cost registers: lines 225 us instead of 211)
            build(std::integral_constant<int, 2>{});
        if (todo >= 1)
            build(std::integral_constant<int, 1>{});
        __syncwarp();
        const bool mine0 = vis.key[0] >= 0 && run[0] >= first && run[0] < first + n;
        const bool mine1 = vis.key[1] >= 0 && run[1] >= first && run[1] < first + n;
        float2 x[2];
        sum_step<COMP, false>(x, ws.slot[(start + (mine0 ? run[0] - first : 0)) & (kSlots - 1)],
                              ws.slot[(start + (mine1 ? run[1] - first : 0)) & (kSlots - 1)], st, lane);
        if (mine0)
            V[0] = x[0];
        if (mine1)
            V[1] = x[1];
        __syncwarp();                   // slots read before the next round builds into them
    }
}

// SMALL: by pieces, without a chunk table.
template <int DT, bool COMP, bool SMALL>
__global__ void __launch_bounds__(kMaxWarps * kWarp, 2)
degrid_kernel(const Geometry g, const void *__restrict__ subgrids, const float *__restrict__ scale,
              const double *__restrict__ uvw, const float *__restrict__ guv,
              const float *__restrict__ gwt, const Schedule sched, float2 *__restrict__ vis_out,
              DeviceStatus *__restrict__ status, const bool vec_ok, const bool prefetch_uvw, const Pieces pieces)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // [w table (optional)] [one WarpSmem per warp]
    WarpSmem &ws = reinterpret_cast<WarpSmem *>(smem_raw + wtable_bytes(g))[threadIdx.x >> 5];
    const float4 *wtab = load_wtable(g, gwt, smem_raw);
    const int lane = threadIdx.x & 31;
    const BuildArgs A{subgrids, wtab, gwt, vec_ok, lane};

    // coordinates in device memory are prefetched into L2 a chunk ahead;
    // coordinates read in place from host memory are not (the host link
    // bounds those calls, and one batch of lead hides its latency)
    pdl_wait();                         // the chunk table is complete
    const auto claimer = [&] {
        if constexpr (SMALL)
            return PieceClaimerT<kStepVis>(pieces, lane);
        else
            return ClaimerT<kStepVis>(sched, lane, Prefetch{prefetch_uvw ? uvw : nullptr, 3 * (int)sizeof(double),
                                                            nullptr, 0});
    };
    Steps<decltype(claimer())> steps{claimer(), uvw + 3 * lane, vis_out + lane};
    const bool checks = SMALL && blockIdx.x == 0 && threadIdx.x < kWarp;
    Step pA = steps.claim();            // the step being summed
    if (pA.n == 0) {
        if (checks)
            check_offsets(pieces, status, lane);
        return;
    }
    Coords3 c[2];
    load_coords(c, pA, lane);
    Vis2 vA = snap_step(pA, c, g, status, lane);
    copy_rows(ws.st, vA, guv, lane);
    Step pB = steps.advance(pA);        // the step after it, its coordinates in registers
    load_coords(c, pB, lane);

    MCache mc{-2, -1, 0};
    int m_s = -1;
    int64_t base = 0;
    float sc = 1.f;
    while (true) {
        const Vis2 vB = snap_step(pB, c, g, status, lane);
        const Step pC = steps.advance(pB);
        load_coords(c, pC, lane);

        if (pA.s != m_s) {
            m_s = pA.s;
            mc.key = -2;
            base = (int64_t)pA.s * g.plane;
            if (DT != DG_C64)
                sc = __ldg(scale + pA.s);
        }
        cp_async_wait<0>();
        __syncwarp();                   // every lane's copies
        float2 V[2];
        if (__all_sync(kFull, vA.key[0] == mc.key && vA.fw[0] == mc.fw && vA.key[1] == mc.key && vA.fw[1] == mc.fw))
            // the whole step continues the cached run (nearly always, on dense lists)
            sum_step<COMP, true>(V, ws.slot[mc.slot], ws.slot[mc.slot], ws.st, lane);
        else
            sum_runs<DT, COMP>(V, mc, ws, ws.st, base, vA, g, A);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (DT != DG_C64)
                V[h] = __fmul2_rn(V[h], make_float2(sc, sc));
            if (lane + kBatch * h < pA.n)
                pA.out[kBatch * h] = V[h];
        }
        if (pB.n == 0)
            break;
        __syncwarp();                   // the rows have been read
        copy_rows(ws.st, vB, guv, lane);
        vA = vB;
        pA = pB;
        pB = pC;
    }
    if (checks)
        check_offsets(pieces, status, lane);
}

size_t smem_bytes(const degrid_plan *p, int warps)
{
    return wtable_bytes_host(p->geo) + sizeof(WarpSmem) * (size_t)warps;
}

// Dynamic shared memory opened so far for a kernel instance on a device.
template <int DT, bool COMP, bool SMALL>
std::atomic<size_t> &smem_record(int device)
{
    static std::atomic<size_t> table[kMaxDevices];
    return dg_smem_record(table, device);
}

template <int DT, bool COMP, bool SMALL>
cudaError_t launch(degrid_plan *p, cudaStream_t st, const void *subgrids, const float *scale,
                   const double *uvw, float2 *out, const Schedule &sched, const Pieces &pieces, int grid_blocks)
{
    const int threads = p->warps_per_block * kWarp;
    const size_t smem = smem_bytes(p, p->warps_per_block);
    cudaError_t e = dg_open_smem(smem_record<DT, COMP, SMALL>(p->device), degrid_kernel<DT, COMP, SMALL>,
                                 smem);
    if (e != cudaSuccess)
        return e;
    // 16-byte footprint loads need an aligned stack and nz a multiple of the
    // elements per 16 bytes
    const bool vec_ok = (reinterpret_cast<uintptr_t>(subgrids) & 15) == 0 &&
                        p->geo.nz % Storage<DT>::kQuad == 0;
    return launch_pdl(degrid_kernel<DT, COMP, SMALL>, dim3(grid_blocks), dim3(threads), smem, st,
                      p->geo, subgrids, scale, uvw, (const float *)p->guv, (const float *)p->gw, sched, out,
                      p->status, vec_ok, !p->host_inputs, pieces);
}

template <int DT, bool COMP, bool SMALL>
int max_blocks(degrid_plan *p)
{
    int n = 0;
    const size_t smem = smem_bytes(p, p->warps_per_block);
    if (dg_open_smem(smem_record<DT, COMP, SMALL>(p->device), degrid_kernel<DT, COMP, SMALL>, smem) !=
        cudaSuccess)
        return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, degrid_kernel<DT, COMP, SMALL>,
                                                      p->warps_per_block * kWarp, smem) != cudaSuccess)
        return 1;
    return n > 0 ? n : 1;
}

// Kernel instance of a plan: storage type and compensated reduction.  Plans
// with a 2D G_uv table (table2d.cu) or with the direct arm (direct.cu) have
// kernels of their own.
template <int DT>
cudaError_t launch_dt(degrid_plan *p, cudaStream_t st, const void *subgrids, const float *scale,
                      const double *uvw, float2 *out, const Schedule &sched, const Pieces &pieces, int grid_blocks)
{
    const auto run = [&](auto fn) { return fn(p, st, subgrids, scale, uvw, out, sched, pieces, grid_blocks); };
    if (pieces.per_warp > 0)
        return p->compensated ? run(launch<DT, true, true>) : run(launch<DT, false, true>);
    return p->compensated ? run(launch<DT, true, false>) : run(launch<DT, false, false>);
}

template <int DT>
int max_blocks_dt(degrid_plan *p)
{
    return p->compensated ? max_blocks<DT, true, false>(p) : max_blocks<DT, false, false>(p);
}

}  // namespace
}  // namespace dg

cudaError_t dg_launch_degrid(degrid_plan *p, cudaStream_t st, const void *subgrids,
                             const float *scale, const double *uvw, const dg::Pieces &pieces,
                             float *out_f, int grid_blocks)
{
    using namespace dg;
    if (p->guv2)
        return dg_launch_degrid_2d(p, st, subgrids, scale, uvw, out_f, grid_blocks);
    if (p->direct_runs < DG_DIRECT_RUNS_NEVER)
        return dg_launch_degrid_direct(p, st, subgrids, scale, uvw, out_f, grid_blocks);
    Schedule sched{p->chunks, p->n_chunks, p->work_counter};
    float2 *out = reinterpret_cast<float2 *>(out_f);
    switch (p->dtype) {
    case DG_C64:
        return launch_dt<DG_C64>(p, st, subgrids, scale, uvw, out, sched, pieces, grid_blocks);
    case DG_C32_F16:
        return launch_dt<DG_C32_F16>(p, st, subgrids, scale, uvw, out, sched, pieces, grid_blocks);
    case DG_C32_BF16:
        return launch_dt<DG_C32_BF16>(p, st, subgrids, scale, uvw, out, sched, pieces, grid_blocks);
    }
    return cudaErrorInvalidValue;
}

int dg_max_blocks_per_sm_degrid(degrid_plan *p)
{
    using namespace dg;
    if (p->guv2)
        return dg_max_blocks_per_sm_degrid_2d(p);
    if (p->direct_runs < DG_DIRECT_RUNS_NEVER)
        return dg_max_blocks_per_sm_degrid_direct(p);
    switch (p->dtype) {
    case DG_C64: return max_blocks_dt<DG_C64>(p);
    case DG_C32_F16: return max_blocks_dt<DG_C32_F16>(p);
    case DG_C32_BF16: return max_blocks_dt<DG_C32_BF16>(p);
    }
    return 1;
}

int dg_max_warps_per_block() { return dg::kMaxWarps; }
