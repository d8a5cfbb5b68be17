// ia_fixed.cuh -- correctly rounded operations of the initial-condition sampler on the integer pipes.
//
// An FP64 instruction occupies a sub-partition of this GPU for 64-76 cycles; a 64 x 64 -> 64-bit high
// product takes about 22 (four 32-bit multiply-adds and the carries). A double square root or division is
// a dozen FP64 instructions; here both are Newton iterations in 64-bit fixed point from the FP32 hardware
// seed, about 100 cycles, run beside the FP64 unit. The result is the correctly rounded one, bit for bit
// what sqrt() and / return: the iterations are good to 2^-60, a 53-bit square root or quotient is never
// exactly between two doubles, and where the eleven bits below the result lie too close to that middle, or
// the operands are not ordinary numbers, the FP64 operation decides.
#pragma once

#include <cstdint>

namespace ia_sample {

typedef unsigned long long u64;
typedef long long i64;

// Positive number m 2^(e - 64), m in [2^63, 2^64).
struct Fx {
    u64 m;
    int e;
};

__device__ __forceinline__ u64 mulhi(u64 a, u64 b) { return __umul64hi(a, b); }

// Sign and value to the nearest double (ties upward); the exponent must be in the normal range.
__device__ __forceinline__ double fx_double(Fx x, bool neg)
{
    // (m >> 11) carries the implicit bit, which adds one to the exponent field; so does a carry of rounding
    const u64 b = ((u64)(x.e + 1021) << 52) + (x.m >> 11) + ((x.m >> 10) & 1ull);
    return __longlong_as_double((i64)(b | (neg ? 0x8000000000000000ull : 0ull)));
}

// Positive normal double.
__device__ __forceinline__ Fx fx_from(double d)
{
    const u64 b = (u64)__double_as_longlong(d);
    Fx r;
    r.m = (b << 11) | 0x8000000000000000ull;
    r.e = (int)(b >> 52) - 1022;
    return r;
}

__device__ __forceinline__ Fx fx_norm(u64 m, int e)
{
    const int s = __clzll((i64)m);
    Fx r;
    r.m = m << s;
    r.e = e - s;
    return r;
}

// Uniform ((x >> 11) | 1) 2^-53: the odd integer times 2^-53, exactly.
__device__ __forceinline__ u64 uniform_int(u64 x) { return (x >> 11) | 1ull; }
__device__ __forceinline__ double uniform_double(u64 k)
{
    return fx_double(fx_norm(k, 11), false);
}

// Square root: m 2^-64 shifted into [1/4, 1) by an even exponent.
__device__ __forceinline__ Fx fx_sqrt(Fx v)
{
    const int odd = v.e & 1;
    const u64 m = odd ? v.m >> 1 : v.m;    // v = (m 2^-64) 2^(e + odd)
    const float wf = __uint2float_rz((unsigned)(m >> 32)) * 0x1p-32f;
    const float yf = rsqrtf(wf);
    const unsigned s0 = __float2uint_rz(fminf(wf * yf, 0x1.fffffep-1f) * 0x1p32f);
    const unsigned Y = __float2uint_rz(fminf(yf, 0x1.fffffep0f) * 0x1p31f);
    i64 d = (i64)(m - (u64)s0 * s0);       // |d| < 2^44: s0 is off by 2^-21 at most
    u64 s = ((u64)s0 << 32) + (u64)(((d >> 14) * (i64)Y) >> 18);
    s = (s >> 63) || (s >> 62) == 1ull ? s : ~0ull;  // the step may pass 1
    d = (i64)(m - mulhi(s, s));            // s is off by 2^-41 at most
    const u64 r = s + (u64)((d * (i64)Y) >> 32);
    Fx o;
    // rounding may leave [1/2, 1) by a unit at either end
    o.m = (r >> 63) ? r : ((r >> 62) ? 1ull << 63 : ~0ull);
    o.e = (v.e + odd) >> 1;
    return o;
}


// True when the bits below the 53rd are within 16 units of the middle between two doubles (or of nothing:
// an exact result rounds the same from either side).
__device__ __forceinline__ bool near_middle(u64 m)
{
    return (unsigned)((m & 0x7ffull) - (0x400ull - 16ull)) <= 32u;
}

__device__ __forceinline__ bool ordinary(double x)  // positive, exponent within 2^+-500
{
    const unsigned hi = (unsigned)__double2hiint(x);
    return hi - ((1023u - 500u) << 20) < (1000u << 20);
}

// sqrt(x), x >= 0.
__device__ __forceinline__ double sqrt_rn(double x)
{
    if (ordinary(x)) {
        const Fx r = fx_sqrt(fx_from(x));
        if (!near_middle(r.m)) return fx_double(r, false);
    }
    return sqrt(x);
}

// 1 / b to 2^-61, b ordinary.
__device__ __forceinline__ Fx fx_rcp(double b)
{
    const Fx v = fx_from(b);               // w = v.m 2^-64 in [1/2, 1)
    const float yf = __frcp_rn(__uint2float_rz((unsigned)(v.m >> 32)) * 0x1p-32f);
    const unsigned Y = __float2uint_rz(fminf(yf, 0x1.fffffep0f) * 0x1p31f);
    u64 y = (u64)Y << 31;                  // 2^62 scale, in (1, 2]
    i64 d = (i64)((1ull << 62) - mulhi(v.m, y));   // 1 - w y, 2^62 scale, below 2^40
    y += (u64)(((d >> 9) * (i64)Y) >> 22);
    d = (i64)((1ull << 62) - mulhi(v.m, y));
    y += (u64)((d * (i64)Y) >> 31);
    return fx_norm(y, 2 - v.e);
}

// a / b given r = 1 / b, b ordinary.
__device__ __forceinline__ double div_rn(double a, double b, Fx r)
{
    if (ordinary(fabs(a))) {
        const Fx x = fx_from(fabs(a));
        const u64 p = mulhi(x.m, r.m);
        const bool top = (p >> 63) != 0ull;
        Fx q;
        q.m = top ? p : p << 1;
        q.e = x.e + r.e - (top ? 0 : 1);
        if (!near_middle(q.m)) return fx_double(q, a < 0.0);
    }
    return a / b;
}

}  // namespace ia_sample
