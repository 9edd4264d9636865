// The subgrid producer's fused transform (predict.cu), for the sizes listed
// in predict_fft.cu.
//
// An item is four planes: of one subgrid (its last item may have fewer), or,
// where a subgrid has one or two, of four or two subgrids.  Per pass of items:
//   rows_kernel     screen and row transforms: image -> work buffer
//   columns_kernel  column transforms, cell window, interleaved stores
// so the planes cross memory once each way between them (the screen, library
// transform and window kernels this replaced moved them four times each way).
//
// Both kernels keep R points of a line per thread in registers and exchange
// them through shared memory between two radices (fft.cuh).  The centred
// transform needs no signs: input and output indices are shifted by N / 2.
// Work layout: [item][kx / 4][row][kx mod 4][plane]: a tile of four columns
// and four planes is contiguous, 128 bytes per image row, so the row kernel
// writes and the column kernel reads whole 128-byte lines, and the column
// kernel stores four cells x four planes (128 bytes of the stack) at once.
//
// Measured on 64 subgrids of 512 x 512 x 4: 653 -> 355 us a call (21 of
// 384 x 384 x 4: 239 -> 92 us); with 1, 2, 3, 5 and 7 planes 287 -> 165, 427
// -> 262, 576 -> 385, 917 -> 831 and 1240 -> 997 us; 64 of 200 x 200 x 3 148
// -> 88 us.  Of each 32 subgrids the row kernel takes 97
// us at 44% of the issue slots (51 instructions per point, 31 of them FP32),
// the column kernel 87 us at 6.2 TB/s of DRAM traffic.
#pragma once

#include "fft.cuh"
#include "internal.cuh"

namespace dg {
namespace {

constexpr int kItemPlanes = 4;                  // planes per item
constexpr int kTileCols = 4;                    // columns per tile of the work buffer
constexpr int kRowPair = 2;                     // image rows per block of the row kernel
constexpr int kRowLines = kRowPair * kItemPlanes;
constexpr int kColLines = kTileCols * kItemPlanes;

// exp(-2 pi i w (n - 1)) with w = (w_hi + w_lo) and n - 1 = (n_hi + n_lo):
// the turns of the product are reduced to [-1/2, 1/2] in double-float
// arithmetic (|w (n - 1)| < 2^22 turns), then rotated in FP32.
__device__ __forceinline__ float2 screen_phasor(float w_hi, float w_lo, float2 nm)
{
    const float p = w_hi * nm.x;
    const float e = fmaf(w_hi, nm.x, -p);                   // p + e = w_hi * n_hi exactly
    const float c = fmaf(w_hi, nm.y, w_lo * nm.x);          // cross terms (w_lo * n_lo dropped)
    const float f = (p - rintf(p)) + (e + c);               // p - rint(p) is exact
    float s, co;
    sincospif(2.0f * f, &s, &co);
    return make_float2(co, -s);
}

__device__ __forceinline__ float2 screen_phasor(double w, float2 nm)
{
    const float hi = (float)w;
    return screen_phasor(hi, (float)(w - (double)hi), nm);
}

template <class F>
struct RowsShape {
    static constexpr int kThreads = kRowLines * F::T;
    static constexpr int kPitch = (F::N + 15) / 16 * 16;           // places of a line's input: whole bank lines
    static constexpr int kExchange = kPitch * kRowLines;           // float2
    // At N = 512 this is 56 KB, which is what four blocks per SM leave each.
    static constexpr size_t kSmem = sizeof(float2) * (kExchange + kRowPair * F::N * 3);
    static constexpr int kBySmem = (int)((size_t)228 * 1024 / (kSmem + 1024));
    static constexpr int kByRegs = 65536 / (kThreads * (F::R > 32 ? 168 : F::R > 16 ? 128 : 96));
    static constexpr int kBlocks = kBySmem < 1 || kByRegs < 1 ? 1 : kBySmem < kByRegs ? kBySmem : kByRegs;
    // Place of transform index n of a line in the exchange: a first-stage
    // butterfly's results are radix(0) places apart, so every other butterfly
    // trades neighbours and two of them fill a 128-byte bank line.
    static_assert(F::radix(0) % 2 == 0, "pairs of places stay within a butterfly");
    __device__ __forceinline__ static int place(int n, int line)
    {
        return (n ^ (n / F::radix(0) & 1)) * kRowLines + line;
    }
    // Place of pixel x of image line `line` (the transform's input): the
    // eight lines of a warp's read start in the four 32-byte bank groups.
    __device__ __forceinline__ static int input_place(int x, int line)
    {
        return line * kPitch + (x ^ ((line & 3) << 2));
    }
};

template <class F>
struct ColumnsShape {
    static constexpr int kThreads = kColLines * F::T;
    static constexpr int kTile = F::N * kColLines;                          // float2: a tile of the work buffer
    static constexpr int kExchange = kTile + F::N / F::radix(0) * kColLines;    // floats, one 64-byte step per first-stage butterfly
    static constexpr size_t kSmem = sizeof(float2) * kTile + sizeof(float) * kExchange;
    static constexpr int kBySmem = (int)((size_t)225 * 1024 / (kSmem + 1024));
    static constexpr int kByRegs = 65536 / (kThreads * (F::R > 32 ? 168 : F::R > 16 ? 128 : 80));
    static constexpr int kBlocks = kBySmem < 1 || kByRegs < 1 ? 1 : kBySmem < kByRegs ? kBySmem : kByRegs;
};

// What a pass works on: subgrids [first, first + n) of nz planes as `count`
// items.
struct PassItems {
    int first, n, nz;
    int count;
    int groups;             // items per subgrid (not PACKED)
    // Subgrid and plane of plane c of item it < count; none if not held(s, p).
    // PACKED: nz is 1 or 2 and items run over the subgrids' planes.
    template <bool PACKED>
    __device__ __forceinline__ void plane(int it, int c, int &s, int &p) const
    {
        if (PACKED) {
            const int q = it * kItemPlanes + c;
            s = nz == 1 ? q : q >> 1;
            p = nz == 1 ? 0 : q & 1;
        } else {
            s = it / groups;
            p = (it - s * groups) * kItemPlanes + c;
        }
        s += first;
    }
    __device__ __forceinline__ bool held(int s, int p) const { return s < first + n && p < nz; }
};

// Screen and row transforms.  A unit is two image rows of one item (eight
// lines); a block takes a contiguous range of units ordered by row pair, so
// it keeps a row pair's tapered image, n - 1 and the plane step's screen in
// shared memory over many items.  The phase of the first plane that an item
// has of a subgrid is computed per pixel, and turned by the plane step for the
// planes after it.  (One instance for both kinds of item ran 5% slower with
// four planes per subgrid, 377 against 356 us on 64 subgrids of 512 x 512;
// three planes per subgrid as PACKED items 474 us against 385, for the parts
// of sectors that the column kernel then stores.)
template <class F, bool PACKED>
__global__ void __launch_bounds__(RowsShape<F>::kThreads, RowsShape<F>::kBlocks)
rows_kernel(const float2 *__restrict__ image, const float *__restrict__ taper, const float2 *__restrict__ nm1,
            const double *__restrict__ w_planes, PassItems items, const float2 *__restrict__ tw,
            float2 *__restrict__ work, bool first_pass)
{
    using Shape = RowsShape<F>;
    constexpr int N = F::N, R = F::R, T = F::T, kThreads = Shape::kThreads;
    constexpr int kImage = kRowPair * N, kPixels = (kImage + kThreads - 1) / kThreads;
    const auto mine = [](int i) { return kImage % kThreads == 0 || i < kImage; };      // pixel i is one of the pair's
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float2 *ex = reinterpret_cast<float2 *>(smem_raw);             // the lines' input, then their exchange
    float2 *base = ex + Shape::kExchange;                           // [row][N]: tapered image
    float2 *nm = base + kRowPair * N;                               // [row][N]: n - 1
    float2 *step = nm + kRowPair * N;                               // [row][N]: the plane step's screen
    const int tid = threadIdx.x;
    // lane = plane + 4 row + 8 (t mod 4): a warp stores 256 contiguous bytes
    const int line = tid & (kRowLines - 1), c = line & 3, row = line >> 2, t = tid / kRowLines;
    pdl_trigger();
    if (first_pass)
        pdl_wait();                     // the n - 1 table is complete
    const long long units = (long long)(N / kRowPair) * items.count;
    const int u_end = (int)(units * (blockIdx.x + 1) / gridDim.x);
    int pair = -1;
    bool have_step = false, waited = first_pass;
    double step_dw = 0.0;
    for (int u = (int)(units * blockIdx.x / gridDim.x); u < u_end; ++u) {
        const int up = u / items.count, item = u - up * items.count;
        // base, nm and step are read and written by the same thread only
        if (up != pair) {
            pair = up;
            have_step = false;
#pragma unroll
            for (int j = 0; j < kPixels; ++j) {
                const int i = tid + j * kThreads, r = i / N, x = i - r * N;
                if (!mine(i))
                    break;
                const int a = x < N / 2 ? x + N / 2 : x - N / 2;    // pixel of transform index x
                const int y = kRowPair * up + r;
                const int b = y < N / 2 ? y + N / 2 : y - N / 2;
                const int da = a < N / 2 ? N / 2 - a : a - N / 2, db = b < N / 2 ? N / 2 - b : b - N / 2;
                float2 m = nm1[db * (N / 2 + 1) + da];
                float2 v = make_float2(0.f, 0.f);
                if (isnan(m.x)) {
                    m = make_float2(0.f, 0.f);
                } else {
                    v = image[b * N + a];
                    const float tp = taper ? taper[b * N + a] : 1.f;
                    v = make_float2(v.x * tp, v.y * tp);
                }
                base[i] = v;
                nm[i] = m;
            }
        }
        if constexpr (!PACKED) {
            int s, plane;
            items.plane<false>(item, 0, s, plane);
            const double dw = w_planes[2 * s + 1], w = w_planes[2 * s] + (double)plane * dw;
            if (!have_step || dw != step_dw) {
#pragma unroll
                for (int j = 0; j < kPixels; ++j)
                    if (mine(tid + j * kThreads))
                        step[tid + j * kThreads] = screen_phasor(dw, nm[tid + j * kThreads]);
                have_step = true;
                step_dw = dw;
            }
            __syncthreads();            // the previous unit's exchange has been read
            const float w_hi = (float)w, w_lo = (float)(w - (double)w_hi);
#pragma unroll
            for (int j = 0; j < kPixels; ++j) {
                const int i = tid + j * kThreads, r = i / N, x = i - r * N;
                if (!mine(i))
                    break;
                float2 cur = cmul(base[i], screen_phasor(w_hi, w_lo, nm[i]));
                const float2 st = step[i];
#pragma unroll
                for (int p = 0; p < kItemPlanes; ++p) {
                    ex[Shape::input_place(x, kItemPlanes * r + p)] = cur;
                    cur = cmul(cur, st);
                }
            }
        } else {
            __syncthreads();            // the previous unit's exchange has been read
            float2 cur[kPixels];
            int last = -1;
#pragma unroll
            for (int p = 0; p < kItemPlanes; ++p) {
                int s, plane;
                items.plane<true>(item, p, s, plane);
                if (!items.held(s, plane)) {                    // past the last plane: nobody stores it
#pragma unroll
                    for (int j = 0; j < kPixels; ++j)
                        cur[j] = make_float2(0.f, 0.f);
                } else if (s == last) {
#pragma unroll
                    for (int j = 0; j < kPixels; ++j)
                        if (mine(tid + j * kThreads))
                            cur[j] = cmul(cur[j], step[tid + j * kThreads]);
                } else {
                    last = s;
                    const double dw = w_planes[2 * s + 1], w = w_planes[2 * s] + (double)plane * dw;
                    if (p + 1 < kItemPlanes && plane + 1 < items.nz && (!have_step || dw != step_dw)) {
#pragma unroll
                        for (int j = 0; j < kPixels; ++j)
                            if (mine(tid + j * kThreads))
                                step[tid + j * kThreads] = screen_phasor(dw, nm[tid + j * kThreads]);
                        have_step = true;
                        step_dw = dw;
                    }
                    const float w_hi = (float)w, w_lo = (float)(w - (double)w_hi);
#pragma unroll
                    for (int j = 0; j < kPixels; ++j)
                        if (mine(tid + j * kThreads))
                            cur[j] = cmul(base[tid + j * kThreads], screen_phasor(w_hi, w_lo, nm[tid + j * kThreads]));
                }
#pragma unroll
                for (int j = 0; j < kPixels; ++j) {
                    const int i = tid + j * kThreads, r = i / N, x = i - r * N;
                    if (mine(i))
                        ex[Shape::input_place(x, kItemPlanes * r + p)] = cur[j];
                }
            }
        }
        __syncthreads();
        float2 v[R];
#pragma unroll
        for (int k = 0; k < R; ++k)
            v[k] = ex[Shape::input_place(t + T * k, line)];
        F::template stage<0>(v, tw, t);
        static_for<F::kStages - 1>([&](auto is) {
            constexpr int S = decltype(is)::value;
            __syncthreads();            // what ex held has been read
            F::template results<S>(v, t, [&](int n, float2 x) { ex[Shape::place(n, line)] = x; });
            __syncthreads();
#pragma unroll
            for (int k = 0; k < R; ++k)
                v[k] = ex[Shape::place(t + T * k, line)];
            F::template stage<S + 1>(v, tw, t);
        });
        if (!waited) {
            pdl_wait();                 // the column kernel of the previous pass has read the buffer
            waited = true;
        }
        // column kx = t + T k of image row y: tile kx / 4, 128 bytes per row
        float2 *dst = work + ((size_t)item * (N / kTileCols) + t / kTileCols) * (N * kColLines) +
                      (kRowPair * up + row) * kColLines + (t % kTileCols) * kItemPlanes + c;
#pragma unroll
        for (int k = 0; k < R; ++k)
            __stcg(dst + (size_t)k * (T / kTileCols) * (N * kColLines), v[k]);
    }
}

// A streaming store under a predicate: a branch around a thread's stores would
// hold them back until the last of its results (1.2% of a call).
__device__ __forceinline__ void store_if(bool yes, float2 *p, float2 v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %0, 0;\n\t@q st.global.cs.v2.f32 [%1], {%2, %3};\n\t}"
                 ::"r"((int)yes), "l"(p), "f"(v.x), "f"(v.y)
                 : "memory");
}

// Column transforms of the tiles of a pass, and the cell window: cell x of
// subgrid s is column (x - N/2 + u0) mod N, cell y likewise.  A block works
// through tiles; the next tile, one contiguous piece of the work buffer, is
// copied into shared memory (cp.async) while the current one is transformed.
// The exchange moves real and imaginary parts one after the other, so both
// fit: two blocks per SM at N = 512.
template <class F, bool PACKED>
__global__ void __launch_bounds__(ColumnsShape<F>::kThreads, ColumnsShape<F>::kBlocks)
columns_kernel(const float2 *__restrict__ work, const int32_t *__restrict__ uv_offsets, PassItems items,
               const float2 *__restrict__ tw, float2 *__restrict__ sub_out)
{
    constexpr int N = F::N, R = F::R, T = F::T, kThreads = ColumnsShape<F>::kThreads;
    constexpr int kTile = ColumnsShape<F>::kTile;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float2 *in = reinterpret_cast<float2 *>(smem_raw);
    float *ex = reinterpret_cast<float *>(in + kTile);
    const int tid = threadIdx.x;
    const int line = tid & (kColLines - 1), c = line & 3, col = line >> 2, t = tid / kColLines;
    const auto fetch = [&](int tile) {
        const float4 *src = reinterpret_cast<const float4 *>(work + (size_t)tile * kTile);
        const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(in));
#pragma unroll
        for (int i = 0; i < kTile / 2 / kThreads; ++i)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * (tid + i * kThreads)),
                         "l"(src + tid + i * kThreads)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    static_assert(kTile / 2 % kThreads == 0, "whole 16-byte copies per thread");
    const int tiles = items.count * (N / kTileCols);
    pdl_trigger();
    pdl_wait();                         // the row kernel's buffer is complete
    if (blockIdx.x < tiles)
        fetch(blockIdx.x);
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int it = tile / (N / kTileCols), kx = (tile - it * (N / kTileCols)) * kTileCols + col;
        // this lane's plane, and its offsets reduced to [0, N): cell = index
        // + N/2 - offset (mod N)
        int s, plane, cx = 0, cy = 0;
        items.plane<PACKED>(it, c, s, plane);
        const bool stored = items.held(s, plane);
        if (stored) {
            cx = (N / 2 - uv_offsets[2 * s] % N) % N;
            cy = (N / 2 - uv_offsets[2 * s + 1] % N) % N;
            cx += cx < 0 ? N : 0;
            cy += cy < 0 ? N : 0;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                // the tile has landed; the last exchange has been read
        float2 v[R];
#pragma unroll
        for (int k = 0; k < R; ++k)
            v[k] = in[(t + T * k) * kColLines + line];
        F::template stage<0>(v, tw, t);
        static_for<F::kStages - 1>([&](auto is) {
            constexpr int S = decltype(is)::value;
            const auto at = [&](int n) { return (n + n / F::radix(0)) * kColLines + line; };
            if (S > 0)
                __syncthreads();        // imaginary parts of the last exchange have been read
            F::template results<S>(v, t, [&](int n, float2 x) { ex[at(n)] = x.x; });
            __syncthreads();            // (the tile has been read, too)
            if (S == 0 && tile + gridDim.x < tiles)
                fetch(tile + gridDim.x);
            float re[R];
#pragma unroll
            for (int k = 0; k < R; ++k)
                re[k] = ex[at(t + T * k)];
            __syncthreads();
            F::template results<S>(v, t, [&](int n, float2 x) { ex[at(n)] = x.y; });
            __syncthreads();
#pragma unroll
            for (int k = 0; k < R; ++k)
                v[k] = make_float2(re[k], ex[at(t + T * k)]);
            F::template stage<S + 1>(v, tw, t);
        });
        const int x = kx + cx < N ? kx + cx : kx + cx - N;
        const int pitch = N * items.nz; // elements per subgrid stay below 2^31
        float2 *dst = sub_out + (size_t)s * N * pitch + (size_t)x * items.nz + plane;
        // rows t + cy + T k until they wrap, the rest N rows up
        float2 *up = dst + (ptrdiff_t)(t + cy - N) * pitch;
        dst += (ptrdiff_t)(t + cy) * pitch;
        const int wrap = (N - t - cy + T - 1) / T;
#pragma unroll
        for (int k = 0; k < R; ++k)
            store_if(stored, (k < wrap ? dst : up) + k * (T * pitch), v[k]);
    }
}

}  // namespace
}  // namespace dg
