// Host side of the producer's fused transform (predict_fft.cuh): which sizes
// it covers, its tables and work buffer, and the passes of a call.
#include <math.h>

#include <new>
#include <vector>

#include "predict_fft.cuh"
#include "predict_fft.h"

namespace dg {
namespace {

// n - 1 of the pixel |a - N/2|, |b - N/2| pixels off the centre, in the
// cancellation-free form -r^2 / (1 + sqrt(1 - r^2)), as the unevaluated sum
// hi + lo of two floats; hi NaN outside the unit circle.  It depends on the
// two distances only, so one quadrant [N/2 + 1][N/2 + 1] serves the image,
// and a thread with x <= y fills both (x, y) and (y, x): FP64 square roots
// and divisions run at a small fraction of the FP32 rate.
__global__ void nm1_quadrant_kernel(float2 *__restrict__ nm1, int half, double dl)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x > y)
        return;
    const double l = (double)x * dl, m = (double)y * dl;
    const double r2 = l * l + m * m;
    float2 v = make_float2(__int_as_float(0x7fc00000), 0.f);
    if (r2 < 1.0) {
        const double d = -r2 / (1.0 + sqrt(1.0 - r2));
        const float hi = (float)d;
        v = make_float2(hi, (float)(d - (double)hi));
    }
    nm1[y * (half + 1) + x] = v;
    nm1[x * (half + 1) + y] = v;
}

}  // namespace
}  // namespace dg

struct dg_predict_fft {
    int n, nz;                      // side; planes per subgrid
    int pass;                       // subgrids per pass at most
    int blocks_rows, blocks_cols;   // resident blocks on the device
    float2 *work, *nm1, *tw;
    const struct Variant *v;
};

namespace {

using namespace dg;

struct RowsArgs {
    const float2 *image;
    const float *taper;
    const double *w_planes;
    PassItems items;
    bool first_pass;
};

struct ColumnsArgs {
    const int32_t *uv_offsets;
    PassItems items;
    float2 *out;
};

}  // namespace

// One image size: its kernels and the twiddle table they read.
struct Variant {
    int n;
    cudaError_t (*prepare)(dg_predict_fft *p, int device, int sm_count);
    cudaError_t (*rows)(const dg_predict_fft *p, cudaStream_t st, int blocks, const RowsArgs &a);
    cudaError_t (*columns)(const dg_predict_fft *p, cudaStream_t st, int blocks, const ColumnsArgs &a);
};

namespace {

template <class F>
std::vector<float2> twiddle_table()
{
    std::vector<float2> h((size_t)F::table_size());
    for (int s = 1; s < F::kStages; ++s) {
        const int r = F::radix(s), Ns = F::span(s);
        for (int q = 0; q < F::R / r; ++q)
            for (int m = 1; m < r; ++m)
                for (int t = 0; t < F::T; ++t) {
                    const int j = (t + F::T * q) % Ns;
                    h[(size_t)F::offset(s) + (size_t)(q * (r - 1) + m - 1) * F::T + t] =
                        make_float2((float)cos_turn((m * j) % (Ns * r), Ns * r), (float)-sin_turn((m * j) % (Ns * r), Ns * r));
                }
    }
    return h;
}

template <class F, bool PACKED>
cudaError_t prepare(dg_predict_fft *p, int device, int sm_count)
{
    static_assert(F::T % kTileCols == 0, "a thread's columns share their place in the tiles");
    static std::atomic<size_t> rows_smem[kMaxDevices], cols_smem[kMaxDevices];
    cudaError_t e = dg_open_smem(dg_smem_record(rows_smem, device), rows_kernel<F, PACKED>, RowsShape<F>::kSmem);
    if (e == cudaSuccess)
        e = dg_open_smem(dg_smem_record(cols_smem, device), columns_kernel<F, PACKED>, ColumnsShape<F>::kSmem);
    int nr = 0, nc = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nr, rows_kernel<F, PACKED>, RowsShape<F>::kThreads,
                                                          RowsShape<F>::kSmem);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nc, columns_kernel<F, PACKED>, ColumnsShape<F>::kThreads,
                                                          ColumnsShape<F>::kSmem);
    if (e != cudaSuccess)
        return e;
    p->blocks_rows = (nr > 0 ? nr : 1) * sm_count;
    p->blocks_cols = (nc > 0 ? nc : 1) * sm_count;
    const std::vector<float2> h = twiddle_table<F>();
    e = cudaMalloc((void **)&p->tw, sizeof(float2) * (h.size() + 1));
    if (e == cudaSuccess)
        e = cudaMemcpy(p->tw, h.data(), sizeof(float2) * h.size(), cudaMemcpyHostToDevice);
    return e;
}

template <class F, bool PACKED>
cudaError_t rows(const dg_predict_fft *p, cudaStream_t st, int blocks, const RowsArgs &a)
{
    return launch_pdl(rows_kernel<F, PACKED>, dim3(blocks), dim3(RowsShape<F>::kThreads), RowsShape<F>::kSmem, st, a.image,
                      a.taper, (const float2 *)p->nm1, a.w_planes, a.items, (const float2 *)p->tw, p->work,
                      a.first_pass);
}

template <class F, bool PACKED>
cudaError_t columns(const dg_predict_fft *p, cudaStream_t st, int blocks, const ColumnsArgs &a)
{
    return launch_pdl(columns_kernel<F, PACKED>, dim3(blocks), dim3(ColumnsShape<F>::kThreads), ColumnsShape<F>::kSmem, st,
                      (const float2 *)p->work, a.uv_offsets, a.items, (const float2 *)p->tw, a.out);
}

template <class F, bool PACKED>
constexpr Variant variant()
{
    return Variant{F::N, prepare<F, PACKED>, rows<F, PACKED>, columns<F, PACKED>};
}

// <side, points per thread, radices>: few exchanges (two radices, so one,
// where the registers allow) and enough threads to fill an SM.  Measured: 512
// as (32, 16) 355 us, as (16, 16, 2) 441, as (8, 8, 8) 472 for 64 subgrids of
// four planes; 384 as (24, 4, 4) 91 us, (8, 8, 6) 99, (24, 16) with 48 points
// per thread 116 for 21 subgrids.
// PACKED: for one or two planes per subgrid.
template <bool PACKED>
constexpr Variant kVariants[] = {
    variant<LineFft<64, 8, 8, 8>, PACKED>(), variant<LineFft<96, 24, 24, 4>, PACKED>(),
    variant<LineFft<128, 16, 16, 8>, PACKED>(), variant<LineFft<192, 24, 24, 8>, PACKED>(),
    variant<LineFft<200, 10, 10, 10, 2>, PACKED>(), variant<LineFft<256, 16, 16, 16>, PACKED>(),
    variant<LineFft<320, 40, 40, 8>, PACKED>(), variant<LineFft<384, 24, 24, 4, 4>, PACKED>(),
    variant<LineFft<400, 20, 20, 20>, PACKED>(), variant<LineFft<512, 32, 32, 16>, PACKED>(),
    variant<LineFft<768, 24, 24, 8, 4>, PACKED>(), variant<LineFft<1024, 32, 32, 32>, PACKED>(),
};

template <bool PACKED>
const Variant *find(int n)
{
    for (const Variant &v : kVariants<PACKED>)
        if (v.n == n)
            return &v;
    return nullptr;
}

bool packed(int nz) { return nz <= 2; }

int items_of(int subgrids, int nz)
{
    return packed(nz) ? (subgrids * nz + kItemPlanes - 1) / kItemPlanes
                      : subgrids * ((nz + kItemPlanes - 1) / kItemPlanes);
}

size_t item_bytes(int n) { return sizeof(float2) * (size_t)n * n * kItemPlanes; }

// Most bytes of work buffer a pass uses.  Large passes win although the
// buffer then goes through DRAM: 64 subgrids of 512 x 512 x 4 took 432 us in
// passes of 7 (59 MB, within L2), 397 us of 14 and 372 us of 32 (268 MB), a
// fill, a drain and a row set-up per pass against 1.07 GB of traffic.  More
// gained nothing.
constexpr size_t kPassBytes = size_t(300) << 20;

// Subgrids per pass for S subgrids: at most `most`, chosen by the rounds of
// resident blocks that the two kernels of each pass take (a round of the
// column kernel handles 16 lines per block, one of the row kernel 8, with
// the screen on top) and a fixed cost per pass.
int choose_pass(const dg_predict_fft *p, int S, int most)
{
    const auto cost = [&](int k) {
        const double rows = ceil((double)items_of(k, p->nz) * (p->n / kRowPair) / p->blocks_rows);
        const double cols = ceil((double)items_of(k, p->nz) * (p->n / kTileCols) / p->blocks_cols);
        return (2.8 * rows + 3.7 * cols) * p->n / 512 + 6.0;         // microseconds, roughly
    };
    int best = 1;
    double best_cost = 1e30;
    for (int k = 1; k <= most && k <= S; ++k) {
        const double c = S / k * cost(k) + (S % k ? cost(S % k) : 0.0);
        if (c < best_cost) {
            best_cost = c;
            best = k;
        }
    }
    return best;
}

}  // namespace

bool dg_predict_fft_supported(int n) { return find<true>(n) != nullptr; }

void dg_predict_fft_destroy(dg_predict_fft *p)
{
    if (!p)
        return;
    cudaFree(p->work);
    cudaFree(p->nm1);
    cudaFree(p->tw);
    delete p;
}

cudaError_t dg_predict_fft_create(dg_predict_fft **out, int n, int nz, int per_pass, int device)
{
    *out = nullptr;
    int sm_count = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess)
        return e;
    dg_predict_fft *p = new (std::nothrow) dg_predict_fft();
    if (!p)
        return cudaErrorMemoryAllocation;
    p->n = n;
    p->nz = nz;
    p->v = packed(nz) ? find<true>(n) : find<false>(n);
    const size_t fit = packed(nz) ? kPassBytes / item_bytes(n) * (kItemPlanes / nz) : kPassBytes / (item_bytes(n) * items_of(1, nz));
    p->pass = fit < 1 ? 1 : (size_t)per_pass < fit ? per_pass : (int)fit;
    e = p->v->prepare(p, device, sm_count);
    if (e == cudaSuccess)
        e = cudaMalloc((void **)&p->work, item_bytes(n) * items_of(p->pass, nz));
    if (e == cudaSuccess)
        e = cudaMalloc((void **)&p->nm1, sizeof(float2) * (n / 2 + 1) * (n / 2 + 1));
    if (e != cudaSuccess) {
        dg_predict_fft_destroy(p);
        return e;
    }
    *out = p;
    return cudaSuccess;
}

cudaError_t dg_predict_fft_execute(dg_predict_fft *p, cudaStream_t st, double theta, const float *image,
                                   const float *taper, int n_subgrids, const int32_t *uv_offsets,
                                   const double *w_planes, float *subgrids_out)
{
    const int half = p->n / 2;
    nm1_quadrant_kernel<<<dim3((unsigned)(half / 64 + 1), (unsigned)(half + 1)), 64, 0, st>>>(p->nm1, half,
                                                                                             theta / p->n);
    cudaError_t e = cudaGetLastError();
    const int pass = choose_pass(p, n_subgrids, p->pass);
    for (int first = 0; first < n_subgrids && e == cudaSuccess; first += pass) {
        const int count = n_subgrids - first < pass ? n_subgrids - first : pass;
        const PassItems items{first, count, p->nz, items_of(count, p->nz), items_of(1, p->nz)};
        const int units = items.count * (p->n / kRowPair), tiles = items.count * (p->n / kTileCols);
        const RowsArgs ra{reinterpret_cast<const float2 *>(image), taper, w_planes, items, first == 0};
        e = p->v->rows(p, st, units < p->blocks_rows ? units : p->blocks_rows, ra);
        if (e != cudaSuccess)
            break;
        const ColumnsArgs ca{uv_offsets, items, reinterpret_cast<float2 *>(subgrids_out)};
        e = p->v->columns(p, st, tiles < p->blocks_cols ? tiles : p->blocks_cols, ca);
    }
    return e;
}
