// Khatri-Rao rows as pairs of floats.
//
// GB300 issues 64 FP32 operations for every FP64 one, so the large FP64 Phi
// launches keep their per-element work on the FP32 pipe: an element of a
// Khatri-Rao row is held as 64 bits that are either a pair (hi, lo) of floats
// with value hi + lo (48 and more significant bits), or the element's FP64
// bits with the sign bit set (an "escape"; every value here is >= 0).  The
// pair form holds values within a window around the largest product, scaled
// by a power of two so that the float exponent range covers it; everything
// else -- values a float pair cannot hold with full precision -- escapes and
// is processed in FP64, so no value loses range or precision.
//
// Scales.  Factor m has the exponent k_m (its entries are < 2^k_m, measured
// when a model is set, 0 after a normalisation, whose columns sum to 1) and is
// held as A^(m) 2^(c - k_m) with c = kPairTop / (N - 1) (pair_factor; its escapes hold
// a bound instead of the FP64 bits, which are in A^(m)).  The products of mode
// n are then scaled by 2^K, K = (N - 1) c - sum_{m != n} k_m, and are at most about
// 2^(kPairTop + N - 1).  Pairs hold scaled values in [2^kPairLow, 2^(e_max + 1)).
//
// Layout.  A row holds its columns two by two: hi of column 2v and of 2v + 1, then
// their lo parts, 16 bytes; so a load brings both parts of two columns as the
// operands of packed FP32 instructions.
//
// Error.  A factor pair is rounded to 2^-49 relative at most; a product
// (pair_mul: one exact FP32 product, the two cross products, renormalised)
// adds at most 2^-47, about 1e-15 in the mean.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace cpapr {

constexpr int kPairTop = 60;    // scaled products are about 2^kPairTop at most
constexpr int kPairLow = -80;   // smallest exponent of a pair
constexpr int kPairMax = kPairTop + 7;  // largest exponent of a product pair
constexpr float kPairLowF = 0x1p-80f;

__host__ __device__ constexpr int pair_scale(int nm1) { return kPairTop / nm1; }

__device__ __forceinline__ bool is_escape(float2 p) { return (int)__float_as_uint(p.x) < 0; }

__device__ __forceinline__ float2 escape_of(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) | (1ull << 63);
    return make_float2(__uint_as_float((uint32_t)(b >> 32)), __uint_as_float((uint32_t)b));
}
__device__ __forceinline__ double escape_value(float2 p) {
    const unsigned long long b =
        ((unsigned long long)(__float_as_uint(p.x) & 0x7fffffffu) << 32) | __float_as_uint(p.y);
    return __longlong_as_double((long long)b);
}

// column c of the row of pairs that starts `row` columns into `base`
__device__ __forceinline__ float2 pair_at(const float *base, int64_t row, int c) {
    const float *p = base + 2 * row + 4 * (c >> 1) + (c & 1);
    return make_float2(__ldg(p), __ldg(p + 2));
}

// v 2^s as a pair, or v as an escape where v 2^s lies outside [2^kPairLow, 2^(emax + 1))
__device__ __forceinline__ float2 pair_encode(double v, int s, int emax) {
    if (v == 0.0) return make_float2(0.f, 0.f);
    const int e = (int)((unsigned long long)__double_as_longlong(v) >> 52);  // v >= 0
    const int es = e - 1023 + s;
    if (e == 0 || es < kPairLow || es > emax) return escape_of(v);
    const double w = __hiloint2double(__double2hiint(v) + (s << 20), __double2loint(v));
    const float h = (float)w;
    return make_float2(h, (float)(w - (double)h));
}

// the float f as a double (integer operations; 0 for zero and subnormal f)
__device__ __forceinline__ double df_widen(float f) {
    const uint32_t b = __float_as_uint(f);
    const unsigned long long d = (((unsigned long long)(b & 0x7fffffffu) << 29) + (896ull << 52)) |
                                 ((unsigned long long)(b & 0x80000000u) << 32);
    return (b & 0x7f800000u) ? __longlong_as_double((long long)d) : 0.0;
}

// v 2^s for v >= 0 (an exponent addition where the result is a normal number)
__device__ __forceinline__ double scale_pow2(double v, int s) {
    const int h = __double2hiint(v);
    const int e = (h >> 20) & 0x7ff;
    const int ne = e + s;
    if (e != 0 && e != 2047 && ne > 0 && ne < 2047) return __hiloint2double(h + (s << 20), __double2loint(v));
    return v == 0.0 ? 0.0 : scalbn(v, s);
}

// the element itself (unscaled) in FP64
__device__ __forceinline__ double pair_value(float2 p, int K) {
    if (is_escape(p)) return escape_value(p);
    return scale_pow2(df_widen(p.x) + df_widen(p.y), -K);
}

// v 2^s of a factor's entry: as pair_encode, but an escape's hi is a negative float, its
// magnitude a bound on v 2^s (a power of two not below 2^-126, or infinite), so that
// the magnitude of a product's hi bounds the product to a rounding (2^-20) where
// escapes took part as well (and to 2^-89 where a partial product underflowed).
__device__ __forceinline__ float2 pair_factor(double v, int s, int emax) {
    const float2 p = pair_encode(v, s, emax);
    if (!is_escape(p)) return p;
    const int es = (int)((unsigned long long)__double_as_longlong(v) >> 52) - 1023 + s;
    const uint32_t b = es >= kPairLow ? 0x7f800000u : (uint32_t)(max(es + 1, -126) + 127) << 23;
    return make_float2(__uint_as_float(0x80000000u | b), 0.f);
}

// a b of two pairs (no escapes), renormalised: hi is the sum rounded to nearest
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);  // not to be fused into p + e below
    float e = fmaf(a.x, b.x, -p);
    e = fmaf(a.x, b.y, e);
    e = fmaf(a.y, b.x, e);
    const float h = p + e;
    return make_float2(h, e - (h - p));
}

// Product of the pairs of one element over the gathered factors, in order.
// `mul` is called for every factor after the first; done() tells whether the
// result is a valid pair, exactly zero, or has to be formed in FP64.
// ESC: zero() also where escapes took part (a small one times 0); the Pi build, whose
// escapes take the FP64 product anyway, is 0.3 ms a mode faster without (4-way tensor).
template <bool ESC>
struct PairProduct {
    float2 p;
    float hmin, omin;  // smallest hi of the products, of the operands (ESC: of their magnitudes)
    uint32_t sg;       // sign bits of the operands (escapes)
    __device__ __forceinline__ void start(float2 a) {
        p = a;
        hmin = a.x;
        omin = ESC ? fabsf(a.x) : a.x;
        sg = __float_as_uint(a.x);
    }
    __device__ __forceinline__ void mul(float2 a) {
        p = pair_mul(p, a);
        sg |= __float_as_uint(a.x);
        omin = fminf(omin, ESC ? fabsf(a.x) : a.x);
        hmin = fminf(hmin, p.x);
    }
    __device__ __forceinline__ bool pair_ok() const { return (int)sg >= 0 && hmin >= kPairLowF; }
    __device__ __forceinline__ bool zero() const { return (ESC || (int)sg >= 0) && omin == 0.f; }
};

}  // namespace cpapr
