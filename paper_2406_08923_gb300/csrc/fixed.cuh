// fixed.cuh -- sums of products of doubles in 64-bit fixed point.
//
// GB300's FP64 pipe retires 2 multiply-adds per clock and SM, its integer pipe 32 multiply-adds of
// 32 x 32 + 64 bits (mad.wide; measured 28 to 30 with distinct operands).  Four of those make a
// 64 x 64-bit product, so a linear stencil of doubles runs up to four times faster as integers
// when the values of a neighbourhood share one binary scale, and more where sums share products.
//
// A set of values whose largest magnitude has the (biased) exponent E is held as
// q = trunc(v 2^(1082 - E)): |q| < 2^60, and 7 bits below a double's last place at the largest
// value.  Values are stored biased by 2^60, so that they and sums of up to 8 of them are
// unsigned and split into 32-bit limbs for free.  A weight is an unsigned integer 2^28 wh + wl
// with a sign of its own; the weights of a sum add up to at most 2^60.  Sums of products are exact in
// four 64-bit accumulators and are rounded once, to the nearest double, at the end.
//
// Accuracy: what truncating the values and rounding the weights costs is a few units of 2^-60 of
// the scale times the sum of the weights.  A chain of FP64 multiply-adds costs a few roundings,
// 2^-53 each, of the largest TERM (weight times value): a value far below the scale, or a small
// weight, makes the FP64 chain the more exact one.  Callers bound the terms of every output from
// below (each kernel says how) and evaluate in FP64 where they may be small; infinities, NaN and
// exponents near the ends of the range go the same way.
#pragma once

#include <cmath>

#include "common.cuh"

namespace stn {

typedef unsigned long long u64;
typedef unsigned int u32;

constexpr u64 FX_BIAS = 1ull << 60;
constexpr u32 FX_BIAS_HI = 1u << 28;
constexpr u32 FX_FLAG_HI = 1u << 22;  // high word of 2^54 = 2^-6 of the scale
// scales (biased exponents) that convert without meeting denormals or overflow
constexpr int FX_EMIN = 192, FX_EMAX = 1856;
// scales a sum uses: what lies below FX_EMIN is more than 63 bits below them
constexpr int FX_SMIN = FX_EMIN + 64;

// Exponent code of a set of values from the largest high word (sign cleared): 0 only for all
// zeros, 1 for denormals alone, 2047 for infinities and NaN.
__device__ __forceinline__ int fx_code(u32 hmax, bool any) { return hmax >> 20 ? (int)(hmax >> 20) : (any ? 1 : 0); }

// v as a biased integer at scale E >= its own exponent.  A zero shifts past the last bit, as
// E >= FX_EMIN.
__device__ __forceinline__ u64 fx_from_double(double v, int E) {
    const u32 hi = (u32)__double2hiint(v), lo = (u32)__double2loint(v);
    const int d = min(E - (int)((hi >> 20) & 0x7ffu), 63);
    const u64 m = (((u64)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 7 >> d;
    const int s = (int)hi >> 31;
    const u64 q = ((u64)((u32)(m >> 32) ^ (u32)s) << 32) | ((u32)m ^ (u32)s);
    return q + (FX_BIAS + (u64)(u32)(-s));
}

// A biased value (bias a multiple of 2^60) moved to a scale d >= 0 bits coarser, rounded down.
// shr.u64 takes any shift (0 from 64 on).
__device__ __forceinline__ u64 fx_shift(u64 v, u64 bias, int d) {
    u64 a, b;
    asm("shr.u64 %0, %1, %2;" : "=l"(a) : "l"(v), "r"(d));
    asm("shr.u64 %0, %1, %2;" : "=l"(b) : "l"(bias), "r"(d));
    return a + (bias - b);
}

// Nearest double (ties to even) of the integer v times 2^(ex - 1082), for |v| >= 2^32.
__device__ __forceinline__ double fx_to_double(long long v, int ex) {
    const u32 s = (u32)(v >> 63);
    const u64 a = (u64)((v ^ (v >> 63)) - (v >> 63));
    const int n = __clz((int)(u32)(a >> 32)) - 1;  // top bit to bit 62
    const u64 t = a << n;
    // round to 53 bits: bit 10 is the last place kept
    const u64 m = (t + (u64)(0x1ffu + (((u32)t >> 10) & 1u))) >> 10;  // the leading one at bit 52, or 53 after a carry
    // value = m 2^(10 - n) 2^(ex - 1082); the leading one of m adds 1 to the exponent field
    const u32 f = (u32)(ex - n + 2) << 20;
    return __hiloint2double((int)(((u32)(m >> 32) + f) | (s & 0x80000000u)), (int)(u32)m);
}
// Whether fx_to_double may take v.
__device__ __forceinline__ bool fx_big(long long v) { return (u64)(v + (1ll << 32)) >= (2ull << 32); }
// The same for |v| <= 2^32 (exact), ex from FX_SMIN - 104 on.
__device__ __forceinline__ double fx_small_to_double(long long v, int ex) {
    return (double)v * __hiloint2double((ex - 59) << 20, 0);  // 2^(ex - 1082)
}

// Accumulators of sum W s with W = 2^28 wh + wl, s = 2^32 sh + sl (all unsigned).
struct FxAcc {
    u64 hh = 0, m1 = 0, m2 = 1ull << 27, ll = 0;  // m2 starts at half of the last place kept
    FxAcc() = default;
    __device__ __forceinline__ explicit FxAcc(u64 half) : m2(half) {}
    __device__ __forceinline__ void mac(u32 wh, u32 wl, u64 s) {
        const u32 sh = (u32)(s >> 32), sl = (u32)s;
        hh += (u64)wh * sh;
        m1 += (u64)wh * sl;
        m2 += (u64)wl * sh;
        ll += (u64)wl * sl;
    }
    // sum W s / 2^60, rounded, modulo 2^64, less the bias the caller folded into `corr`
    __device__ __forceinline__ long long result(u64 corr) const {
        return (long long)(hh + ((m2 + (m1 >> 4) + (ll >> 32)) >> 28) + corr);
    }
    __device__ __forceinline__ void add(const FxAcc &o) {
        hh += o.hh;
        m1 += o.m1;
        m2 += o.m2;
        ll += o.ll;
    }
    // sum W s / 2^60 as a double times 2^(ex - 1082), for weights of 60 bits whose sum is at most 2^60,
    // up to 12 of them, and sums that may cancel (m2 started at 0): 28 bits below the last place
    // of the integer are kept.  A negative sum is up to 2^-32 of that place short, a zero is exact.
    __device__ __forceinline__ double wide(u64 corr, int ex) const {
        const u64 x = m2 + (m1 >> 4) + (ll >> 32);
        const u64 r = hh + (x >> 28) + corr;
        const u32 s = (u32)((long long)r >> 63);
        u32 a = (u32)(r >> 32) ^ s, b = (u32)r ^ s, c = ((u32)x << 4) ^ s;
#pragma unroll 1
        for (int i = 0; i < 2 && a == 0u; ++i) {  // the leading bit into a (a branch that is rarely taken)
            a = b;
            b = c;
            c = 0u;
            ex -= 32;
        }
        const int n = __clz((int)a);
        const u32 hi = __funnelshift_l(b, a, n), lo = __funnelshift_l(c, b, n);  // leading bit: bit 63
        const u64 m = (((u64)hi << 32 | lo) >> 11) + ((lo >> 10) & 1u);          // bit 52, or 53 after a carry
        const u32 f = a == 0u ? 0u : (u32)(ex - n + 3) << 20;
        return __hiloint2double((int)(((u32)(m >> 32) + f) | (s & 0x80000000u)), (int)(u32)m);
    }
};

// One launch's weights: |value i| is (2^28 wh + wl) 2^(ew - 60); `corr` takes the bias of every sum
// off the result.  The kernels know the signs: a sum with a negative weight enters as 2^61 mult - s,
// the biased negative.
template <int N> struct FxWeights {
    u32 wh[N], wl[N];
    int ew;
    u64 corr;
};
constexpr int FX_EW = 104;  // |ew| at most

// mult[i]: how many values sum i adds (6 at most, |result| < 2^63).  False where fixed point does not
// apply (a weight is not finite, all are zero, or the exponent is out of range).
template <int N> inline bool fx_weights(const double *w, const int *mult, FxWeights<N> &o) {
    double sum = 0.0;
    for (int i = 0; i < N; ++i) sum += std::fabs(w[i]);
    if (!(sum > 0.0) || !std::isfinite(sum)) return false;
    (void)std::frexp(sum, &o.ew);  // sum < 2^ew
    if (o.ew < -FX_EW || o.ew > FX_EW) return false;
    u64 bias = 0;
    for (int i = 0; i < N; ++i) {
        const u64 W = (u64)std::llrint(std::ldexp(std::fabs(w[i]), 60 - o.ew));
        o.wh[i] = (u32)(W >> 28);
        o.wl[i] = (u32)(W & 0xfffffffu);
        bias += W * (u64)mult[i];
    }
    o.corr = 0ull - bias;
    return true;
}

}  // namespace stn
