// Rows in fixed point for the integer Khat products.  Every row l of the three
// Khat^j is an integer row c over one denominator d_l (sum |c| < 2^23), so with
// X in fixed point below a bound on its row, sum_j sum_m c_jlm X^j_m is formed
// from integer sums.  Binary64 rows: 62 bits in two words, both summed exactly in
// 64-bit integers, one rounding at the end.  An entry under 2^-9 of its row's bound
// thus has less than its own 53 bits: the error is relative to the row's largest
// entries, not to each.  (With the low word as binary32, summed by FFMA, N = 6 took 110
// thousand instead of 114 thousand clocks an element and SM, but its error rose from
// 2.2e-16 to 2.9e-16.)  Double-binary32 rows: a 30-bit word summed in 64-bit integers
// and the remainder as binary32.  GB300 issues binary64 multiply-adds at 2 lanes a
// clock and SM, 64-bit integer ones at 13 to 19, binary32 ones at 125.
#pragma once

#include "dw_device.cuh"
#include "poro_internal.h"

namespace poro {

constexpr int POISON = INT32_MIN;  // row scale of a row with a non-finite bound

// Binary64: x = v 2^s with |x| <= 2^30 as a 64-bit integer with 32 fraction
// bits, as two signed words (high, low).  sh0 = 1053 - s, one more than the biased
// exponent of the row's bound.  (Magnitudes below 2^-1022 are not kept.)
__device__ __forceinline__ int2 quantise(double v, int sh0) {
    const int hi = __double2hiint(v);
    const int E = (hi >> 20) & 0x7FF;
    const uint32_t mh = ((uint32_t)hi & 0xFFFFFu) | (E ? 0x100000u : 0u);
    const unsigned long long m = (((unsigned long long)mh << 32) | (uint32_t)__double2loint(v)) << 10;
    const int sh = sh0 - E;
    long long x = (unsigned)sh < 64u ? (long long)(m >> sh) : 0ll;
    x = hi < 0 ? -x : x;
    const int lo = (int)(uint32_t)x;
    return make_int2((int)((x - (long long)lo) >> 32), lo);
}
// scale word of a row from the bound on its entries
__device__ __forceinline__ int row_scale(double bound) {
    const int E = (__double2hiint(bound) >> 20) & 0x7FF;
    return E == 0x7FF ? POISON : E + 1;
}
__device__ __forceinline__ double bound_of(uint32_t bits, double) {
    return __hiloint2double((int)(bits >= 0x7FF00000u ? 0x7FF80000u : bits + 1u), 0);
}

// (hi 2^32 + lo) 2^(-s - 32) as the nearest binary64 (magnitudes below
// 2^-1022 become zero, beyond the range infinity); sh0 = 1053 - s
__device__ __forceinline__ double fixed_to_double(long long hi, uint32_t w0, int sh0) {
    const bool neg = hi < 0;
    unsigned long long h = (unsigned long long)hi;
    if (neg) {
        w0 = 0u - w0;
        h = ~h + (w0 == 0u ? 1ull : 0ull);
    }
    uint32_t w2 = (uint32_t)(h >> 32), w1 = (uint32_t)h;
    int ex = 1086 - (1053 - sh0);  // biased exponent of bit 95, less its leading zeros below
    if (w2 == 0u) {
        w2 = w1;
        w1 = w0;
        w0 = 0u;
        ex -= 32;
    }
    if (w2 == 0u) {
        w2 = w1;
        w1 = w0;
        ex -= 32;
    }
    if (w2 == 0u) return 0.0;
    const int z = __clz((int)w2);
    const uint32_t th = __funnelshift_l(w1, w2, z), tl = __funnelshift_l(w0, w1, z);
    ex -= z;
    unsigned long long m = ((unsigned long long)th << 32) | tl;
    m = (m >> 11) + ((m >> 10) & 1ull);
    if (ex <= 0) return 0.0;
    if (ex >= 2047) m = 0x7FF0000000000000ull;
    else m += (unsigned long long)(ex - 1) << 52;
    return __longlong_as_double((long long)(m | (neg ? 0x8000000000000000ull : 0ull)));
}
// Double-binary32: x = v 2^s with |x| <= 2^29 as the nearest integer of its
// high word and the remainder in binary32.
__device__ __forceinline__ int2 quantise(float2 v, int s) {
    const float f = pow2f(s);
    const int n = __float2int_rn(__fmul_rn(v.x, f));
    const float r = __fmaf_rn(v.x, f, -(float)n);
    return make_int2(n, __float_as_int(__fmaf_rn(v.y, f, r)));
}
// n + r for an integer |n| < 2^53 and a small r, as (h, l)
__device__ __forceinline__ float2 fixed_to_pair(long long n, float r) {
    const float fa = __fmul_rn(small_int_to_float((int)(n >> 31)), 2147483648.0f);
    const float fb = __fmul_rn(small_int_to_float((int)((n >> 9) & 0x3FFFFF)), 512.0f);
    const float fc = small_int_to_float((int)(n & 511));
    const float g = __fadd_rn(fa, fb);
    const float t = __fadd_rn(__fsub_rn(fb, __fsub_rn(g, fa)), fc);
    const float h = __fadd_rn(g, t);  // |t| below the last place of g, or g = 0
    return make_float2(h, __fadd_rn(__fsub_rn(t, __fsub_rn(h, g)), r));
}
__device__ __forceinline__ int row_scale(float bound) {
    return min(max(29 - ((__float_as_int(bound) >> 23) - 126), -126), 126);
}
__device__ __forceinline__ float bound_of(uint32_t bits, float) { return __uint_as_float(bits); }

// one entry's products: acc += c x, for the integer word and what is below it
__device__ __forceinline__ void fixed_mac(int c, int2 x, long long& hi, long long& lo) {
    hi += (long long)c * x.x;
    lo += (long long)c * x.y;
}
__device__ __forceinline__ void fixed_mac(int c, int2 x, long long& hi, float& lo) {
    hi += (long long)c * x.x;
    lo = __fmaf_rn((float)c, __int_as_float(x.y), lo);
}
// the binary64 sum (NaN for a poisoned row)
__device__ __forceinline__ double fixed_sum(long long hi, long long lo, int sc) {
    const double v = fixed_to_double(hi + (lo >> 32), (uint32_t)lo, sc);
    return sc == POISON ? __longlong_as_double(0x7FF8000000000000LL) : v;
}

// the modes of degree block g that a pass with room for `columns` columns
// (direction, mode) of X takes, three columns a mode: all, or equal parts
PORO_HD constexpr int pass_count(int g, int columns) { return (block_size(g) + columns / 3 - 1) / (columns / 3); }
PORO_HD constexpr int pass_modes(int g, int columns) {
    return (block_size(g) + pass_count(g, columns) - 1) / pass_count(g, columns);
}

}  // namespace poro
