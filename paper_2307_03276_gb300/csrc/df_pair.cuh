// Khatri-Rao rows as pairs of floats.
//
// GB300 issues 64 FP32 operations for every FP64 one, so the large FP64 Phi
// launches keep their per-element work on the FP32 pipe: an element of a
// Khatri-Rao row is held as 64 bits that are a pair (hi, lo) of floats with value
// hi + lo (48 and more significant bits), scaled by a power of two so that the float
// exponent range covers a window around the largest product.  (Every value here is
// >= 0.)  An element outside the window is an escape, a negative hi: kLowEscape below
// it, kHighEscape where a factor's entry is above its exponent.  An escape holds no
// value; where one is needed it is formed in FP64 from the factors.
//
// Scales.  Factor m has the exponent k_m (its entries are < 2^k_m, measured
// when a model is set, 0 after a normalisation, whose columns sum to 1) and is
// held as A^(m) 2^(kPairTop - k_m), from 2^kFactorLow up to 2^kPairTop.  Each product
// of two is scaled back by 2^-kPairTop, so products of mode n carry 2^K, K =
// kPairTop - sum_{m != n} k_m, and never exceed 2^kPairTop, nor a partial product
// they were formed from: an element is below the window (2^kPairLow) as soon as a
// factor's entry is below 2^kFactorLow or a partial product below 2^kPairLow.  With
// products left at the scale of all their factors (2^(60 / (N - 1)) each) that was
// not so, and every element with a small factor was formed in FP64 to find out: within
// 20 outer iterations, with 10 to 18% of the elements small, the build of the 3-way
// tensor's rows (1e7 nonzeros, R = 32) grew from 0.58 to 2.8 ms, and a launch that
// forms them in place from 0.83 to 2.5; now the build stays at 0.58 and the launch
// goes from 0.71 to 0.95, for the sums it takes again (pair_resum).
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

constexpr int kPairTop = 60;      // products and factors are at most 2^kPairTop
constexpr int kPairLow = -80;     // smallest exponent of a product's pair
constexpr int kFactorLow = -100;  // and of a factor's (its lo keeps 24 bits)
constexpr float kPairLowF = 0x1p-80f;
constexpr uint32_t kLowEscape = 0x80800000u;   // -2^-126
constexpr uint32_t kHighEscape = 0xff800000u;  // -infinity

__device__ __forceinline__ bool is_escape(float2 p) { return (int)__float_as_uint(p.x) < 0; }

// column c of the row of pairs that starts `row` columns into `base`
__device__ __forceinline__ float2 pair_at(const float *base, int64_t row, int c) {
    const float *p = base + 2 * row + 4 * (c >> 1) + (c & 1);
    return make_float2(__ldg(p), __ldg(p + 2));
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

// a pair's value (unscaled) in FP64
__device__ __forceinline__ double pair_value(float2 p, int K) { return scale_pow2(df_widen(p.x) + df_widen(p.y), -K); }

// v 2^s of a factor's entry
__device__ __forceinline__ float2 pair_factor(double v, int s) {
    if (v == 0.0) return make_float2(0.f, 0.f);
    const int e = (int)((unsigned long long)__double_as_longlong(v) >> 52);  // v >= 0
    const int es = e - 1023 + s;
    if (e == 0 || es < kFactorLow) return make_float2(__uint_as_float(kLowEscape), 0.f);
    if (es > kPairTop) return make_float2(__uint_as_float(kHighEscape), 0.f);
    const double w = __hiloint2double(__double2hiint(v) + (s << 20), __double2loint(v));
    if (w > 0x1p60) return make_float2(__uint_as_float(kHighEscape), 0.f);
    const float h = (float)w;
    return make_float2(h, (float)(w - (double)h));
}
static_assert(kPairTop == 60, "pair_factor's bound, pair_mul's scale");

// a b 2^-kPairTop of two pairs (no escapes), renormalised: hi is the sum rounded to
// nearest.  The product itself is up to 2^(2 kPairTop); it is scaled back exactly
// where the result is a pair.
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
    constexpr float down = 0x1p-60f;
    const float p = __fmul_rn(a.x, b.x);
    float e = fmaf(a.x, b.x, -p);
    e = fmaf(a.x, b.y, e);
    e = fmaf(a.y, b.x, e) * down;
    const float h = fmaf(p, down, e);  // one rounding of p down + e
    return make_float2(h, e - fmaf(-down, p, h));
}

// Product of the pairs of one element over the gathered factors, in order: `mul`
// is called for every factor after the first.  A low escape makes it small, a high one
// infinite or NaN; a factor of exactly zero makes it zero whatever the others are.
// (Partial products only fall: the last one says whether all were pairs.)
struct PairProduct {
    float2 p;
    float omin;   // smallest magnitude of the operands' hi
    uint32_t sg;  // sign bits of the operands (escapes)
    __device__ __forceinline__ void start(float2 a) {
        p = a;
        omin = fabsf(a.x);
        sg = __float_as_uint(a.x);
    }
    __device__ __forceinline__ void mul(float2 a) {
        p = pair_mul(p, a);
        sg |= __float_as_uint(a.x);
        omin = fminf(omin, fabsf(a.x));
    }
    // is p the element?  Else it is value()
    __device__ __forceinline__ bool pair_ok() const { return (int)sg >= 0 && p.x >= kPairLowF; }
    __device__ __forceinline__ bool plain_zero() const { return (int)sg >= 0 && omin == 0.f; }  // p is (0, 0)
    __device__ __forceinline__ bool plain() const { return (int)sg >= 0 && (p.x >= kPairLowF || omin == 0.f); }
    __device__ __forceinline__ float2 value() const {
        if (pair_ok()) return p;
        if (omin == 0.f) return make_float2(0.f, 0.f);
        const bool high = (int)sg < 0 && !(fabsf(p.x) < __int_as_float(0x7f800000));
        return make_float2(__uint_as_float(high ? kHighEscape : kLowEscape), 0.f);
    }
};

}  // namespace cpapr
