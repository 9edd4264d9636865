// Register FFT building blocks: small DFTs on arrays held in registers and
// the stages of a line transform split over several threads.
//
// A line of N points is held by T threads, R = N / T points each: thread t
// holds points t + T k, k = 0 .. R - 1.  A stage of radix r (r divides R)
// is R / r butterflies per thread (Stockham's autosort order): butterfly q,
// j = t + T q, takes points j + m N / r (the thread's own k = q + m R / r),
// multiplies point m by w_{Ns r}^{m (j mod Ns)}, Ns the product of the
// radices before, and leaves its result m at
// (j div Ns) Ns r + j mod Ns + m Ns.  Between two stages the points go
// through shared memory once; the last stage leaves point t + T k in v[k].
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace dg {
namespace {

// ---- compile-time twiddles --------------------------------------------------

constexpr double kPi = 3.14159265358979323846264338327950288;

// cos and sin of x in [0, pi / 4] by their power series.
__host__ __device__ constexpr double cos_small(double x)
{
    double t = 1.0, s = 1.0;
    for (int i = 1; i < 12; ++i) {
        t *= -x * x / ((2 * i - 1) * (2 * i));
        s += t;
    }
    return s;
}

__host__ __device__ constexpr double sin_small(double x)
{
    double t = x, s = x;
    for (int i = 1; i < 12; ++i) {
        t *= -x * x / ((2 * i) * (2 * i + 1));
        s += t;
    }
    return s;
}

// cos(2 pi k / n) for any 0 <= k < n, reduced to the first octant in integers.
__host__ __device__ constexpr double cos_turn(int k, int n)
{
    if (2 * k > n)
        k = n - k;                                  // cos(2 pi - x) = cos x
    if (4 * k > n)
        return -cos_turn(n - 2 * k, 2 * n);         // cos(pi - x) = -cos x
    if (8 * k > n)
        return sin_small(2.0 * kPi * (n - 4 * k) / (4.0 * n));
    return cos_small(2.0 * kPi * k / n);
}

__host__ __device__ constexpr double sin_turn(int k, int n)             // cos(x - pi / 2)
{
    return cos_turn((4 * k + 3 * n) % (4 * n), 4 * n);
}

template <class F, int... I>
__device__ __forceinline__ void static_for_impl(std::integer_sequence<int, I...>, F f)
{
    (f(std::integral_constant<int, I>{}), ...);
}

// f(integral_constant<0>) ... f(integral_constant<N - 1>).
template <int N, class F>
__device__ __forceinline__ void static_for(F f)
{
    static_for_impl(std::make_integer_sequence<int, N>{}, f);
}

// ---- complex arithmetic -----------------------------------------------------

// Scalar additions: the packed forms halve the instructions, but run on half
// of the FP32 lanes and measured slower here (372 against 360 us on 64
// subgrids of 512 x 512 x 4).
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// x exp(-2 pi i K / R) with a compile-time K.
template <int R, int K>
__device__ __forceinline__ float2 mul_root(float2 x)
{
    constexpr int k = K % R;
    if constexpr (k == 0)
        return x;
    else if constexpr (4 * k == R)
        return make_float2(x.y, -x.x);
    else if constexpr (2 * k == R)
        return make_float2(-x.x, -x.y);
    else if constexpr (4 * k == 3 * R)
        return make_float2(-x.y, x.x);
    else {
        constexpr float c = (float)cos_turn(k, R), s = (float)sin_turn(k, R);
        return make_float2(fmaf(x.x, c, x.y * s), fmaf(x.y, c, -x.x * s));
    }
}

// ---- small DFTs: x[k] = sum_n x[n] exp(-2 pi i n k / R), in place ------------

template <int R>
__device__ __forceinline__ void dft(float2 (&x)[R])
{
    if constexpr (R == 1) {
    } else if constexpr (R == 2) {
        const float2 a = x[0];
        x[0] = cadd(a, x[1]);
        x[1] = csub(a, x[1]);
    } else if constexpr (R == 3) {
        constexpr float s3 = (float)sin_turn(1, 3);
        const float2 p = cadd(x[1], x[2]), m = csub(x[1], x[2]);
        const float2 c = __ffma2_rn(p, make_float2(-0.5f, -0.5f), x[0]);
        x[0] = cadd(x[0], p);
        x[1] = make_float2(fmaf(s3, m.y, c.x), fmaf(-s3, m.x, c.y));
        x[2] = make_float2(fmaf(-s3, m.y, c.x), fmaf(s3, m.x, c.y));
    } else if constexpr (R == 4) {
        const float2 a = cadd(x[0], x[2]), b = csub(x[0], x[2]), c = cadd(x[1], x[3]), d = csub(x[1], x[3]);
        x[0] = cadd(a, c);
        x[2] = csub(a, c);
        x[1] = make_float2(b.x + d.y, b.y - d.x);
        x[3] = make_float2(b.x - d.y, b.y + d.x);
    } else if constexpr (R == 5) {
        constexpr float c1 = (float)cos_turn(1, 5), c2 = (float)cos_turn(2, 5);
        constexpr float s1 = (float)sin_turn(1, 5), s2 = (float)sin_turn(2, 5);
        const float2 p1 = cadd(x[1], x[4]), m1 = csub(x[1], x[4]), p2 = cadd(x[2], x[3]), m2 = csub(x[2], x[3]);
        const float2 a = __ffma2_rn(p2, make_float2(c2, c2), __ffma2_rn(p1, make_float2(c1, c1), x[0]));
        const float2 b = __ffma2_rn(p2, make_float2(c1, c1), __ffma2_rn(p1, make_float2(c2, c2), x[0]));
        const float2 d = __ffma2_rn(m2, make_float2(s2, s2), __fmul2_rn(m1, make_float2(s1, s1)));
        const float2 e = __ffma2_rn(m2, make_float2(-s1, -s1), __fmul2_rn(m1, make_float2(s2, s2)));
        x[0] = cadd(x[0], cadd(p1, p2));
        x[1] = make_float2(a.x + d.y, a.y - d.x);
        x[4] = make_float2(a.x - d.y, a.y + d.x);
        x[2] = make_float2(b.x + e.y, b.y - e.x);
        x[3] = make_float2(b.x - e.y, b.y + e.x);
    } else {
        // R = A B: X[k1 + A k2] = sum_b w_R^{b k1} (sum_a x[B a + b] w_A^{a k1}) w_B^{b k2}
        constexpr int A = R % 4 == 0 ? 4 : R % 2 == 0 ? 2 : R % 3 == 0 ? 3 : 5;
        constexpr int B = R / A;
        static_assert(A * B == R && B > 1, "radices 2, 3 and 5 only");
        float2 y[A][B];
        static_for<B>([&](auto ib) {
            constexpr int b = decltype(ib)::value;
            float2 t[A];
#pragma unroll
            for (int a = 0; a < A; ++a)
                t[a] = x[B * a + b];
            dft<A>(t);
            static_for<A>([&](auto ik) {
                constexpr int k1 = decltype(ik)::value;
                y[k1][b] = mul_root<R, b * k1>(t[k1]);
            });
        });
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            dft<B>(y[k1]);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2)
                x[k1 + A * k2] = y[k1][k2];
        }
    }
}

// ---- stages -------------------------------------------------------------------

// A line transform: N points, R per thread, radices in order.
template <int N_, int R_, int... Rad>
struct LineFft {
    static constexpr int N = N_, R = R_, T = N_ / R_;
    static constexpr int kStages = sizeof...(Rad);
    static_assert(T * R == N && (Rad * ... * 1) == N, "the radices make up the line");
    static_assert(((R_ % Rad == 0) && ...), "every radix divides the points per thread");
    __host__ __device__ static constexpr int radix(int s)
    {
        constexpr int r[] = {Rad...};
        return r[s];
    }
    // product of the radices before stage s
    __host__ __device__ static constexpr int span(int s)
    {
        int p = 1;
        for (int i = 0; i < s; ++i)
            p *= radix(i);
        return p;
    }
    // Twiddles of stage s > 0 for butterfly q, point m of thread t are at
    // offset(s) + (q (r - 1) + m - 1) T + t of the table: a constant plus t.
    __host__ __device__ static constexpr int twiddles(int s) { return R / radix(s) * (radix(s) - 1) * T; }
    __host__ __device__ static constexpr int offset(int s)
    {
        int o = 0;
        for (int i = 1; i < s; ++i)
            o += twiddles(i);
        return o;
    }
    __host__ __device__ static constexpr int table_size() { return offset(kStages); }

    // Twiddles and butterflies of stage S (0-based) on this thread's points.
    template <int S>
    __device__ __forceinline__ static void stage(float2 (&v)[R], const float2 *__restrict__ tw, int t)
    {
        constexpr int r = radix(S), Q = R / r;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float2 x[r];
#pragma unroll
            for (int m = 0; m < r; ++m) {
                x[m] = v[q + m * Q];
                if (S > 0 && m > 0)
                    x[m] = cmul(x[m], __ldg(tw + offset(S) + (q * (r - 1) + m - 1) * T + t));
            }
            dft<r>(x);
#pragma unroll
            for (int m = 0; m < r; ++m)
                v[q + m * Q] = x[m];
        }
    }

    // put(n, value) for every result n of stage S.
    template <int S, class F>
    __device__ __forceinline__ static void results(const float2 (&v)[R], int t, F put)
    {
        constexpr int r = radix(S), Q = R / r, Ns = span(S);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int j = t + T * q;
            const int n0 = j / Ns * (Ns * r) + j % Ns;
#pragma unroll
            for (int m = 0; m < r; ++m)
                put(n0 + m * Ns, v[q + m * Q]);
        }
    }
};

}  // namespace
}  // namespace dg
