// In-register FFTs of up to 32 points, one line per thread.
#pragma once

#include "cplx.cuh"

namespace mb {

// Twiddles in the scaled form of the radix-2 butterfly with fused
// multiply-adds (Linzer & Feig, 1993): the twiddle w = cos a + i sin a of
// angle a = 2 pi k / 32 is stored as w = c (1 + i r) with (c, r) = (cos a,
// tan a) where |cos a| >= |sin a|, else as w = c (r + i) with (c, r) =
// (sin a, cot a).  Then a +- w b costs two fused multiply-adds for
// t = b (1 + i r) (or b (r + i)) and four for a +- c t: six per butterfly
// instead of eight for a complex product and two complex additions, with
// |r| <= 1 so that no term is amplified.
constexpr double kC1 = 0.98078528040323044913, kT1 = 0.19891236737965800691;   // cos, tan of pi/16
constexpr double kC2 = 0.92387953251128675613, kT2 = 0.41421356237309504880;   // of pi/8
constexpr double kC3 = 0.83146961230254523708, kT3 = 0.66817863791929891999;   // of 3 pi/16
constexpr double kC4 = 0.70710678118654752440;                                 // of pi/4 (tan = 1)
#define MB_TW32(T)                                                                                          \
    {                                                                                                       \
        {1, 0}, {T(kC1), T(kT1)}, {T(kC2), T(kT2)}, {T(kC3), T(kT3)}, {T(kC4), 1}, {T(kC3), T(kT3)},        \
        {T(kC2), T(kT2)}, {T(kC1), T(kT1)}, {1, 0}, {T(kC1), T(-kT1)}, {T(kC2), T(-kT2)},                   \
        {T(kC3), T(-kT3)}, {T(-kC4), -1}, {T(-kC3), T(-kT3)}, {T(-kC2), T(-kT2)}, {T(-kC1), T(-kT1)}        \
    }
static __constant__ float2 c_tsf[16] = MB_TW32(float);
static __constant__ double2 c_tsd[16] = MB_TW32(double);
#undef MB_TW32

constexpr bool tw_tan_form(int k) { return k <= 4 || k >= 12; }   // k < 16

template <typename C> __device__ __forceinline__ C ctws(int k);
template <> __device__ __forceinline__ float2 ctws<float2>(int k) { return c_tsf[k]; }
template <> __device__ __forceinline__ double2 ctws<double2>(int k) { return c_tsd[k]; }

__device__ __forceinline__ float fmar(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return fma(a, b, c); }

constexpr int brev_c(int x, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((x >> b) & 1) << (bits - 1 - b);
    return r;
}
constexpr int ilog2_c(int n) { return n <= 1 ? 0 : 1 + ilog2_c(n / 2); }

// (a, b) <- (a + w b, a - w b), w = exp(sign 2 pi i tk / N), sign = + for the
// inverse transform (the forward twiddle is the conjugate: r and, in the
// cot form, c change sign)
template <int N, bool INV, typename C>
__device__ __forceinline__ void bfly(C &a, C &b, int tk) {
    const C u = a;
    if (tk == 0) {
        a = u + b;
        b = u - b;
        return;
    }
    if (4 * tk == N) {
        const C wb = INV ? mk(-b.y, b.x) : mk(b.y, -b.x);
        a = u + wb;
        b = u - wb;
        return;
    }
    const int k = tk * (32 / N);
    const C q = ctws<C>(k);
    auto c = q.x, r = q.y;
    const bool tan_form = tw_tan_form(k);
    if (!INV) {
        r = -r;
        if (!tan_form) c = -c;
    }
    C t;
    if (tan_form) {
        t.x = fmar(-r, b.y, b.x);
        t.y = fmar(r, b.x, b.y);
    } else {
        t.x = fmar(r, b.x, -b.y);
        t.y = fmar(r, b.y, b.x);
    }
    a.x = fmar(c, t.x, u.x);
    a.y = fmar(c, t.y, u.y);
    b.x = fmar(-c, t.x, u.x);
    b.y = fmar(-c, t.y, u.y);
}

// true when every input index that reaches positions [p, p + len) of the
// bit-reversed array is >= nin (those positions hold zeros until the stage
// that merges them with a lower block)
constexpr bool zero_block(int p, int len, int bits, int nin) {
    for (int i = p; i < p + len; ++i)
        if (brev_c(i, bits) < nin) return false;
    return true;
}
// bit q: the lower half of butterfly group q of the stage of half-width
// `half` is all zeros
constexpr unsigned long long stage_zero_mask(int n, int half, int bits, int nin) {
    unsigned long long m = 0;
    for (int g = 0; g < n; g += 2 * half)
        if (nin < n && zero_block(g + half, half, bits, nin)) m |= 1ull << (g / (2 * half));
    return m;
}

template <int N, bool INV, int NIN, int HALF, typename C>
__device__ __forceinline__ void fft_stages(C (&x)[N]) {
    constexpr unsigned long long zm = stage_zero_mask(N, HALF, ilog2_c(N), NIN);
#pragma unroll
    for (int g = 0; g < N; g += 2 * HALF) {
#pragma unroll
        for (int j = 0; j < HALF; ++j) {
            if ((zm >> (g / (2 * HALF))) & 1) x[g + j + HALF] = x[g + j];
            else bfly<N, INV>(x[g + j], x[g + j + HALF], j * (N / (2 * HALF)));
        }
    }
    if constexpr (2 * HALF < N) fft_stages<N, INV, NIN, 2 * HALF>(x);
}

// in-register radix-2 FFT of N <= 32 points (natural order in and out);
// inputs NIN .. N-1 are known to be zero, and the butterflies whose lower
// operand is still all zeros become copies (a + w 0 = a - w 0 = a)
template <int N, bool INV, int NIN = N, typename C>
__device__ __forceinline__ void fft_reg(C (&x)[N]) {
    static_assert(N <= 32, "twiddle table of 32nds of a turn");
    constexpr int L = ilog2_c(N);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int j = brev_c(i, L);
        if (j > i) {
            C t = x[i];
            x[i] = x[j];
            x[j] = t;
        }
    }
    fft_stages<N, INV, NIN, 1>(x);
}

}  // namespace mb
