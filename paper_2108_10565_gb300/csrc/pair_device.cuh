// The two arithmetics of Biot's kernels behind one interface: IEEE binary64,
// and double-binary32 pairs on the binary32 pipe (dw_device.cuh).
#pragma once

#include "dw_device.cuh"

namespace poro {

// x as (hi, lo) binary32 words, as dw_split gives them, on the integer pipe
// (dw_split's conversions run on the binary64 pipe): hi is x rounded to 24 bits
// (ties up), lo the rest rounded.  Values whose words leave binary32's normal
// range take dw_split.
__device__ __forceinline__ float2 dw_cut(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int E = (hi >> 20) & 0x7FF;
    if (E < 930 || E > 1140) return x == 0.0 ? make_float2(0.f, 0.f) : dw_split(x);
    const int sg = hi & 0x80000000;
    // the 24 leading bits, rounded up (with the carry into the exponent) when
    // the 29 bits below are at least half, and those bits as what is left
    const int up = (lo >> 28) & 1;
    const float h = __int_as_float(sg | ((((E - 896) << 23) | ((hi & 0xFFFFF) << 3) | (int)((uint32_t)lo >> 29)) + up));
    const int rest = (lo & 0x1FFFFFFF) - (up << 29);  // in units of 2^(E - 1075)
    const float r = (float)rest * __int_as_float(sg | ((E - 1075 + 29 + 127) << 23));
    return make_float2(h, r * 1.862645149230957e-9f);  // 2^-29
}

struct Bin64Base {
    using R = double;
    static constexpr bool DW = false;
    static constexpr uint32_t INF = 0x7FF00000u;  // of the high word
    __device__ static R zero() { return 0.0; }
    __device__ static R of(double x) { return x; }
    __device__ static double value(R a) { return a; }
    __device__ static R mul(R a, R b) { return a * b; }
    __device__ static R fma(R a, R b, R c) { return ::fma(a, b, c); }
    __device__ static R fma1(float k, R b, R c) { return ::fma((double)k, b, c); }
    __device__ static R add(R a, R b) { return a + b; }
    __device__ static R sub(R a, R b) { return a - b; }
    __device__ static R neg(R a) { return -a; }
    __device__ static R shfl(R v, int src) { return __shfl_sync(0xffffffffu, v, src); }
    __device__ static R select(bool c, R a, R b) { return c ? a : b; }
    __device__ static R normal(R a) { return a; }
    __device__ static uint32_t abs_bits(R a) { return (uint32_t)__double2hiint(a) & 0x7FFFFFFFu; }

    // PACK values side by side
    static constexpr int PACK = 1;
    using V = double;
    __device__ static V zeros() { return 0.0; }
    __device__ static V all(R a) { return a; }
    __device__ static V vmul(V a, V b) { return a * b; }
    __device__ static V vfma(V a, V b, V c) { return ::fma(a, b, c); }
    __device__ static V vadd(V a, V b) { return a + b; }
    __device__ static V vsub(V a, V b) { return a - b; }
    __device__ static R sum(V a) { return a; }
};

// the packed binary32 operations: one issue slot for two results
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f32x2 pk_fma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 pk_mul(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 pk_add(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// times -1, which is exact, stands for the sign modifier that the packed forms lack
constexpr f32x2 MINUS_ONES = 0xBF800000BF800000ull;
__device__ __forceinline__ f32x2 pk_neg(f32x2 a) { return pk_mul(a, MINUS_ONES); }
__device__ __forceinline__ f32x2 pk_sub(f32x2 a, f32x2 b) { return pk_fma(b, MINUS_ONES, a); }

// unevaluated sums (x, y) of two binary32 words, about 48 bits
struct Bin32x2Base {
    using R = float2;
    static constexpr bool DW = true;
    static constexpr uint32_t INF = 0x7F800000u;
    __device__ static R zero() { return make_float2(0.f, 0.f); }
    __device__ static R of(double x) { return dw_cut(x); }
    __device__ static double value(R a) { return pair_to_double(a.x, a.y); }  // of a normalised pair
    __device__ static R mul(R a, R b) {
        const float p = __fmul_rn(a.x, b.x);
        return make_float2(p, __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.y, __fmaf_rn(a.x, b.x, -p))));
    }
    __device__ static R fma(R a, R b, R c) {
        dw_mac(c.x, c.y, a.x, a.y, b.x, b.y);
        return c;
    }
    __device__ static R fma1(float k, R b, R c) {
        dw_mac_x2(c.x, c.y, k, b.x, b.y);
        return c;
    }
    __device__ static R add(R a, R b) {
        float s, e;
        two_sum(a.x, b.x, s, e);
        return make_float2(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
    }
    __device__ static R sub(R a, R b) { return add(a, neg(b)); }
    __device__ static R neg(R a) { return make_float2(-a.x, -a.y); }
    __device__ static R shfl(R v, int src) {
        return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
    }
    __device__ static R select(bool c, R a, R b) { return make_float2(c ? a.x : b.x, c ? a.y : b.y); }
    __device__ static R normal(R a) {
        float s, e;
        two_sum(a.x, a.y, s, e);
        return make_float2(s, e);
    }
    __device__ static uint32_t abs_bits(R a) { return __float_as_uint(a.x) & 0x7FFFFFFFu; }

    // two values side by side, both high words, then both low ones; the same
    // operations in the same order as above, bit for bit
    static constexpr int PACK = 2;
    struct __align__(16) V {
        f32x2 h, l;
    };
    __device__ static V zeros() { return {0ull, 0ull}; }
    __device__ static V all(R a) { return {pack2(a.x, a.x), pack2(a.y, a.y)}; }
    __device__ static V vmul(V a, V b) {
        const f32x2 p = pk_mul(a.h, b.h);
        return {p, pk_fma(a.l, b.h, pk_fma(a.h, b.l, pk_fma(a.h, b.h, pk_neg(p))))};
    }
    __device__ static V vfma(V a, V b, V c) {
        const f32x2 p = pk_mul(a.h, b.h);
        const f32x2 e = pk_fma(a.l, b.h, pk_fma(a.h, b.l, pk_fma(a.h, b.h, pk_neg(p))));
        const f32x2 s = pk_add(c.h, p), bb = pk_sub(s, c.h);
        const f32x2 er = pk_add(pk_sub(c.h, pk_sub(s, bb)), pk_sub(p, bb));
        return {s, pk_add(c.l, pk_add(er, e))};
    }
    __device__ static V vadd(V a, V b) {
        const f32x2 s = pk_add(a.h, b.h), bb = pk_sub(s, a.h);
        const f32x2 er = pk_add(pk_sub(a.h, pk_sub(s, bb)), pk_sub(b.h, bb));
        return {s, pk_add(er, pk_add(a.l, b.l))};
    }
    __device__ static V vsub(V a, V b) { return vadd(a, {pk_neg(b.h), pk_neg(b.l)}); }
    __device__ static R sum(V a) {
        const float2 h = unpack2(a.h), l = unpack2(a.l);
        return add(make_float2(h.x, l.x), make_float2(h.y, l.y));
    }
};

}  // namespace poro
