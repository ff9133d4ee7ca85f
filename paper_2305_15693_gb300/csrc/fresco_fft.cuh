// In-place transforms in shared memory (fresco_fft.h describes a transform): the butterflies, the
// passes, the forward transform and its adjoint, shared by the kernels that fuse them with the steps
// around them.
//
// Decimation in frequency forward, which leaves frequency k at place pos[k], and its adjoint,
// decimation in time, back: the steps in between work on the permuted order through a table and no
// pass reorders. The inverse runs on values with real and imaginary part exchanged, which turns it
// into the same butterflies and twiddles as the forward transform. The first pass takes its input
// through a loader and the adjoint's last one leaves its output through a storer (global memory).
// Twiddles: one table value per butterfly, its powers by multiplication (at most four products
// deep). The radix-R butterflies are the plain sums for 3, 5 and 7 (symmetric and antisymmetric
// parts), and two-step splits for the composite ones (Cooley and Tukey 1965).
#pragma once

#include <cuda_runtime.h>

#include "fresco_fft.h"

namespace fresco {

namespace fft_detail {

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return {fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.x, b.y, a.y * b.x)};
}
__device__ __forceinline__ float2 mul_mi(float2 a) { return {a.y, -a.x}; }   // -i a

// cos and sin of 2 pi k / R, k <= (R - 1) / 2 (k is a constant once the loops are unrolled)
template <int R>
__device__ __forceinline__ float root_cos(int k) {
    if (R == 3) return -0.5f;
    if (R == 5) return k == 1 ? 0.30901699437494742410f : -0.80901699437494742410f;
    return k == 1 ? 0.62348980185873353053f
                  : (k == 2 ? -0.22252093395631440429f : -0.90096886790241912624f);
}
template <int R>
__device__ __forceinline__ float root_sin(int k) {
    if (R == 3) return 0.86602540378443864676f;
    if (R == 5) return k == 1 ? 0.95105651629515357212f : 0.58778525229247312917f;
    return k == 1 ? 0.78183148246802980871f
                  : (k == 2 ? 0.97492791218182360702f : 0.43388373911755812048f);
}

template <int R>
struct Dft {   // odd primes
    static __device__ __forceinline__ void run(float2 (&x)[R]) {
        constexpr int H = (R - 1) / 2;
        float2 t[H + 1], u[H + 1];
        float2 sum = x[0];
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            t[k] = cadd(x[k], x[R - k]);
            u[k] = csub(x[k], x[R - k]);
            sum = cadd(sum, t[k]);
        }
        const float2 x0 = x[0];
#pragma unroll
        for (int p = 1; p <= H; ++p) {
            float2 a = x0, b = {0.f, 0.f};
#pragma unroll
            for (int k = 1; k <= H; ++k) {
                const int i = (p * k) % R;
                const float c = root_cos<R>(i <= H ? i : R - i);
                const float s = i <= H ? root_sin<R>(i) : -root_sin<R>(R - i);
                a = {fmaf(c, t[k].x, a.x), fmaf(c, t[k].y, a.y)};
                b = {fmaf(s, u[k].x, b.x), fmaf(s, u[k].y, b.y)};
            }
            x[p] = {a.x + b.y, a.y - b.x};       // a - i b
            x[R - p] = {a.x - b.y, a.y + b.x};   // a + i b
        }
        x[0] = sum;
    }
};
template <>
struct Dft<2> {
    static __device__ __forceinline__ void run(float2 (&x)[2]) {
        const float2 a = x[0], b = x[1];
        x[0] = cadd(a, b);
        x[1] = csub(a, b);
    }
};
template <>
struct Dft<4> {
    static __device__ __forceinline__ void run(float2 (&x)[4]) {
        const float2 a0 = cadd(x[0], x[2]), a1 = csub(x[0], x[2]);
        const float2 a2 = cadd(x[1], x[3]), a3 = mul_mi(csub(x[1], x[3]));
        x[0] = cadd(a0, a2);
        x[2] = csub(a0, a2);
        x[1] = cadd(a1, a3);
        x[3] = csub(a1, a3);
    }
};

// cos and sin of 2 pi k / N at compile time, by their series about 0 on the first octant
struct Unit {
    double c, s;
};
constexpr Unit unit_series(double t) {
    double c = 0.0, s = 0.0, p = 1.0;   // p = t^j / j!
    for (int j = 0; j < 26; ++j) {
        const double sg = (j & 2) ? -1.0 : 1.0;
        if (j & 1) s += sg * p;
        else c += sg * p;
        p *= t / (j + 1);
    }
    return {c, s};
}
constexpr Unit unit_root(int k, int n) {
    // 8 k / n = octant o and remainder
    const int o = 8 * k / n;
    const double q = 6.283185307179586476925286766559 / n;
    const Unit u = (o & 1) ? unit_series(q * ((o + 1) * n / 8.0 - k)) : unit_series(q * (k - o * n / 8.0));
    // the angle is (o + 1) pi / 4 minus, or o pi / 4 plus, the reduced one
    const double r = 0.70710678118654752440084436210485;
    const int b = (o & 1) ? o + 1 : o;
    const double cb[9] = {1, r, 0, -r, -1, -r, 0, r, 1}, sb[9] = {0, r, 1, r, 0, -r, -1, -r, 0};
    const double sg = (o & 1) ? -1.0 : 1.0;
    return {cb[b] * u.c - sg * sb[b] * u.s, sb[b] * u.c + sg * cb[b] * u.s};
}

// a exp(-2 pi i K / N) for the two-step splits
template <int N, int K>
__device__ __forceinline__ float2 twiddle_const(float2 a) {
    if constexpr (K == 0) return a;
    else if constexpr (4 * K == N) return mul_mi(a);
    else if constexpr (2 * K == N) return {-a.x, -a.y};
    else {
        constexpr Unit u = unit_root(K % N, N);
        constexpr float c = (float)u.c, s = (float)-u.s;
        return cmul(a, {c, s});
    }
}

// N = A B: x[B a + b]; transforms over a, twiddles, transforms over b; result p1 + A p2
template <int A, int B>
struct DftAB {
    static constexpr int N = A * B;
    template <int BB, int P>
    static __device__ __forceinline__ void twiddle(float2 (&y)[B][A]) {
        if constexpr (P < A) {
            y[BB][P] = twiddle_const<N, BB * P>(y[BB][P]);
            twiddle<BB, P + 1>(y);
        } else if constexpr (BB + 1 < B) {
            twiddle<BB + 1, 0>(y);
        }
    }
    static __device__ __forceinline__ void run(float2 (&x)[N]) {
        float2 y[B][A];
#pragma unroll
        for (int b = 0; b < B; ++b) {
#pragma unroll
            for (int a = 0; a < A; ++a) y[b][a] = x[B * a + b];
            Dft<A>::run(y[b]);
        }
        twiddle<0, 0>(y);
#pragma unroll
        for (int p = 0; p < A; ++p) {
            float2 z[B];
#pragma unroll
            for (int b = 0; b < B; ++b) z[b] = y[b][p];
            Dft<B>::run(z);
#pragma unroll
            for (int b = 0; b < B; ++b) x[p + A * b] = z[b];
        }
    }
};
template <> struct Dft<6> : DftAB<3, 2> {};
template <> struct Dft<8> : DftAB<4, 2> {};
template <> struct Dft<9> : DftAB<3, 3> {};
template <> struct Dft<10> : DftAB<5, 2> {};

// x[p] *= w^p
template <int R>
__device__ __forceinline__ void powers(float2 (&x)[R], float2 w) {
    float2 w2 = cmul(w, w);
    x[1] = cmul(x[1], w);
    if constexpr (R > 2) x[2] = cmul(x[2], w2);
    if constexpr (R > 3) {
        float2 pw[R];
        pw[1] = w;
        pw[2] = w2;
#pragma unroll
        for (int p = 3; p < R; ++p) {
            pw[p] = (p & 1) ? cmul(pw[p - 1], w) : cmul(pw[p / 2], pw[p / 2]);
            x[p] = cmul(x[p], pw[p]);
        }
    }
}

// One pass over `rows` transforms. Forward (decimation in frequency): butterfly, then twiddles;
// DIT: twiddles, then butterfly. ld(row, i) and st(row, i, v) reach element i of a row.
template <int R, bool DIT, class Ld, class St>
__device__ __forceinline__ void fft_pass(const FftDesc &f, int p, int rows, Ld ld, St st) {
    const int m = f.m[p], nb = f.n / R, step = nb / m;   // step = n / (m R): twiddle stride
    const int total = rows * nb;
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int row = rows == 1 ? 0 : f.db[p].div(i);
        const int ii = i - row * nb;
        const int blk = f.dm[p].div(ii), j = ii - blk * m;
        const int base = blk * m * R + j;
        float2 x[R];
#pragma unroll
        for (int q = 0; q < R; ++q) x[q] = ld(row, base + q * m);
        if (!DIT) Dft<R>::run(x);
        if (m > 1) powers<R>(x, __ldg(f.tw + j * step));
        if (DIT) Dft<R>::run(x);
#pragma unroll
        for (int q = 0; q < R; ++q) st(row, base + q * m, x[q]);
    }
}

template <bool DIT, class Ld, class St>
__device__ __forceinline__ void fft_pass_any(const FftDesc &f, int p, int rows, Ld ld, St st) {
    switch (f.r[p]) {
#define FRESCO_FFT_CASE(R) case R: fft_pass<R, DIT>(f, p, rows, ld, st); break;
        FRESCO_FFT_CASE(2) FRESCO_FFT_CASE(3) FRESCO_FFT_CASE(4) FRESCO_FFT_CASE(5)
        FRESCO_FFT_CASE(6) FRESCO_FFT_CASE(7) FRESCO_FFT_CASE(8) FRESCO_FFT_CASE(9)
        FRESCO_FFT_CASE(10)
#undef FRESCO_FFT_CASE
        default: break;
    }
}

// Forward transform of rows whose first pass reads through ld; the result is in s (pitch elements a
// row), frequency k at fft_place(pos[k]). Ends with a barrier.
template <class Ld>
__device__ __forceinline__ void fft_forward(const FftDesc &f, int rows, float2 *s, int pitch, Ld ld) {
    auto sl = [&](int row, int i) { return s[row * pitch + fft_place(f, i)]; };
    auto ss = [&](int row, int i, float2 v) { s[row * pitch + fft_place(f, i)] = v; };
    fft_pass_any<false>(f, 0, rows, ld, ss);
    __syncthreads();
    for (int p = 1; p < f.np; ++p) {
        fft_pass_any<false>(f, p, rows, sl, ss);
        __syncthreads();
    }
}

// Adjoint of the above on s (parts exchanged, see the header); the last pass stores through st
// (natural order). Begins after a barrier of the caller.
template <class St>
__device__ __forceinline__ void fft_adjoint(const FftDesc &f, int rows, float2 *s, int pitch, St st) {
    auto sl = [&](int row, int i) { return s[row * pitch + fft_place(f, i)]; };
    auto ss = [&](int row, int i, float2 v) { s[row * pitch + fft_place(f, i)] = v; };
    for (int p = f.np - 1; p > 0; --p) {
        fft_pass_any<true>(f, p, rows, sl, ss);
        __syncthreads();
    }
    fft_pass_any<true>(f, 0, rows, sl, st);
}

}  // namespace fft_detail

}  // namespace fresco
