// Weighted sums of FP64 numbers on the integer pipe, for kernels that stream vectors: with GB300's 2 FP64
// multiply-adds per clock and SM they take longer than the numbers' bytes.  Numbers become 58-bit words under a
// common exponent, weights 57-bit words; products run as in hop_fx.cuh (three integer multiply-adds each), and
// the sum is rounded once.  The words are as long as 8 products in a 64-bit sum allow.
#pragma once

#include "hop_fx.cuh"

// digits of a weight of magnitude up to 2^e: w = (h 2^28 + l) 2^(e - 57)
struct FxWeight {
    int h, l;
};
__device__ inline FxWeight fx_weight(double w, int e) {
    const long long t = (long long)rint(ldexp(w, 57 - e)) + (1ll << 27);
    return FxWeight{(int)(t >> 28), (int)(t & 0x0fffffff) - (1 << 27)};
}
// exponents of the weights and biased exponents of the numbers that are taken: every scale factor and result is
// then a normal number
constexpr int FXW_EXP = 100;
constexpr int FXV_MIN = 200, FXV_MAX = 1800;

// v_j, j < K <= 8, under one exponent: (h_j 2^28 + l_j) 2^(e - 58).  false (nothing set) if the largest is
// zero, very small, very large or not finite: the caller then sums in FP64.
template <int K>
__device__ __forceinline__ bool fx_numbers(const double v[K], int h[K], int l[K], int &e) {
    int mx = 0;
#pragma unroll
    for (int j = 0; j < K; j++) mx = max(mx, __double2hiint(v[j]) & 0x7fffffff);
    const int ef = mx >> 20;
    if (ef < FXV_MIN || ef > FXV_MAX) return false;
    e = ef - 1022;
#pragma unroll
    for (int j = 0; j < K; j++) {
        const int hw = __double2hiint(v[j]);
        const int r = min(ef - (hw >> 20 & 0x7ff), 63);  // a zero's or subnormal's bits are shifted out
        const unsigned long long w = ((unsigned long long)(unsigned)((hw & 0xfffff) | 0x100000) << 38 |
                                      (unsigned long long)(unsigned)__double2loint(v[j]) << 6) >> r;
        const long long sg = (long long)(hw >> 31);
        const long long t = ((long long)w ^ sg) + ((1ll + (1ll << 28)) - sg);  // +- w, rounded to 58 bits, digits split
        h[j] = (int)(t >> 29);
        l[j] = (int)((unsigned)t >> 1 & 0x0fffffff) - (1 << 27);
    }
    return true;
}

// sum_j w_j v_j in units of 2^(e_w + e - FX_SUM_BITS); |sum| <= K 2^59
constexpr int FX_SUM_BITS = 57 + 58 - 2 * 28;
template <int K>
__device__ __forceinline__ long long fx_sum(const FxWeight *w, const int h[K], const int l[K]) {
    long long x = 1ll << 27, y = 0;
#pragma unroll
    for (int j = 0; j < K; j++) {
        x += (long long)w[j].h * l[j];
        x += (long long)w[j].l * h[j];
        y += (long long)w[j].h * h[j];
    }
    return y + (x >> 28);
}
// a 2^ea + b 2^eb in units of 2^e, e the larger exponent; |a|, |b| <= 2^62, |a| + |b| < 2^63
__device__ __forceinline__ long long fx_add(long long a, int ea, long long b, int eb, int &e) {
    e = max(ea, eb);
    const int sa = min(e - ea, 62), sb = min(e - eb, 62);
    return ((a + ((1ll << sa) >> 1)) >> sa) + ((b + ((1ll << sb) >> 1)) >> sb);
}
// v 2^k without an FP64 multiplication (the result is a normal number or zero)
__device__ __forceinline__ double fx_value(long long v, int k) {
    const double d = (double)v;
    return __hiloint2double(v ? __double2hiint(d) + (k << 20) : 0, __double2loint(d));
}
