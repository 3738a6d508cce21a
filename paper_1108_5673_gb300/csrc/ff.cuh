// Float-float arithmetic on the FP32 pipe for the amplitude generators: an
// unevaluated sum h + l of two floats carries ~44 bits at 4 to 16 FP32
// operations a step, where this part's FP64 pipe has 1/64 of the FP32 rate.
// The building blocks are Dekker's and Knuth's error-free sum and the product
// split by FMA (Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26 (2005)). Every
// value is a pair of events in packed FP32 (f2), so that one instruction
// serves both.
//
// Error model, relative to the operands' sizes: a product of normalised pairs
// (|l| <= 2^-24 |h|) 2^-45.4 (the dropped l l' and the two roundings of the low
// part), 2^-44.5 with one operand that is not (|l| <= 2^-22 |h|), 2^-43.7 with
// both; a sum 2^-46.4 of |a| + |b|; a b +- c d 2^-44.5 of |a b| + |c d|; the
// reciprocal and the square root 2^-45. Products of the high parts must stay
// above 2^-100 in size for the split to be exact; the callers check their
// results against thresholds that ensure it.
#pragma once

#include "pwa_internal.cuh"

namespace pwa {

__device__ __forceinline__ f2 neg2(f2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f2 abs2(f2 a) { return a & 0x7fffffff7fffffffull; }
__device__ __forceinline__ f2 dup2(float a) { return pk2(a, a); }

struct ff {
    f2 h, l;
};

__device__ __forceinline__ ff ff_dup(float h, float l) { return {dup2(h), dup2(l)}; }
// a literal as a float pair, rounded at compile time
__device__ __forceinline__ ff ff_const(double x)
{
    return ff_dup((float)x, (float)(x - (double)(float)x));
}

// |a| >= |b| or a = 0: a + b exactly as h + l
__device__ __forceinline__ ff ff_fast(f2 a, f2 b)
{
    const f2 s = add2(a, b);
    return {s, sub2(b, sub2(s, a))};
}

__device__ __forceinline__ ff ff_two_sum(f2 a, f2 b)
{
    const f2 s = add2(a, b), t = sub2(s, a);
    return {s, add2(sub2(a, sub2(s, t)), sub2(b, t))};
}

__device__ __forceinline__ ff ff_two_diff(f2 a, f2 b)
{
    const f2 s = sub2(a, b), t = sub2(s, a);
    return {s, sub2(sub2(a, sub2(s, t)), add2(b, t))};
}

// a b, not renormalised (|l| a few 2^-23 |h|)
__device__ __forceinline__ ff ff_mul(ff a, ff b)
{
    const f2 p = mul2(a.h, b.h);
    f2 e = fma2(a.h, b.h, neg2(p));
    e = fma2(a.h, b.l, e);
    return {p, fma2(a.l, b.h, e)};
}

__device__ __forceinline__ ff ff_mul(ff a, f2 b)
{
    const f2 p = mul2(a.h, b);
    return {p, fma2(a.l, b, fma2(a.h, b, neg2(p)))};
}

__device__ __forceinline__ ff ff_sqr(ff a)
{
    const f2 p = mul2(a.h, a.h);
    return {p, fma2(add2(a.h, a.h), a.l, fma2(a.h, a.h, neg2(p)))};
}

__device__ __forceinline__ ff ff_add(ff a, ff b)
{
    const ff s = ff_two_sum(a.h, b.h);
    return ff_fast(s.h, add2(s.l, add2(a.l, b.l)));
}

__device__ __forceinline__ ff ff_sub(ff a, ff b)
{
    const ff s = ff_two_diff(a.h, b.h);
    return ff_fast(s.h, add2(s.l, sub2(a.l, b.l)));
}

__device__ __forceinline__ ff ff_neg(ff a) { return {neg2(a.h), neg2(a.l)}; }
__device__ __forceinline__ ff ff_norm(ff a) { return ff_fast(a.h, a.l); }

// a b - c d and a b + c d: the products' high parts summed exactly. Not
// renormalised: after cancellation |l| is small against |a b| + |c d| only.
__device__ __forceinline__ ff ff_det(ff a, ff b, ff c, ff d)
{
    const ff x = ff_mul(a, b), y = ff_mul(c, d);
    const ff s = ff_two_diff(x.h, y.h);
    return {s.h, add2(s.l, sub2(x.l, y.l))};
}
__device__ __forceinline__ ff ff_dot(ff a, ff b, ff c, ff d)
{
    const ff x = ff_mul(a, b), y = ff_mul(c, d);
    const ff s = ff_two_sum(x.h, y.h);
    return {s.h, add2(s.l, add2(x.l, y.l))};
}

// 1 / a: a hardware approximation (relative error below 2^-21) and one
// Newton step whose remainder is kept as the low part
__device__ __forceinline__ ff ff_rcp(ff a)
{
    float a0, a1;
    upk2(a.h, a0, a1);
    const f2 r = pk2(rcp_approx(a0), rcp_approx(a1));
    const f2 nr = neg2(r);
    f2 t = fma2(a.h, nr, dup2(1.0f));
    t = fma2(a.l, nr, t);
    return {r, mul2(r, fma2(t, t, t))};
}

// sqrt(a) for a >= 2^-60
__device__ __forceinline__ ff ff_sqrt(ff a)
{
    float a0, a1;
    upk2(a.h, a0, a1);
    const float s0 = sqrtf(a0), s1 = sqrtf(a1);
    const f2 s = pk2(s0, s1);
    const f2 e = add2(fma2(s, neg2(s), a.h), a.l);
    return ff_fast(s, mul2(e, pk2(0.5f / s0, 0.5f / s1)));
}

// d as a float pair, through its bits (conversions of doubles run at the
// FP64 pipe's rate): 24 bits truncated, the other 29 rounded to a float;
// relative error below 2^-47. `ok` is cleared where |d| is outside [2^-60,
// 2^61) and not zero.
__device__ __forceinline__ float2 split_bits(double d, bool &ok)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const int e = (int)((hi >> 20) & 0x7ff);
    const unsigned sign = hi & 0x80000000u;
    const bool in = (unsigned)(e - 963) <= 120u;
    ok = ok && (in || ((hi & 0x7fffffffu) | lo) == 0u);
    const float h = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
    const float unit = __uint_as_float(sign | ((unsigned)(e - 948) << 23));  // 2^(e - 1075)
    const float l = (float)(lo & 0x1fffffffu) * unit;
    return in ? make_float2(h, l) : make_float2(0.f, 0.f);
}

// one double per event to a float pair, renormalised
__device__ __forceinline__ ff ff_split(double d0, double d1, bool &ok0, bool &ok1)
{
    const float2 a = split_bits(d0, ok0), b = split_bits(d1, ok1);
    return ff_fast(pk2(a.x, b.x), pk2(a.y, b.y));
}

// The floats nearest to v, given |v - (a.h + a.l)| <= err: sure where every
// value of that interval rounds to the same float, of at least 2^-70 in size
// (smaller values and zeros, whose low parts may have underflowed, are left
// to the caller). a need not be normalised: the rounding of l +- err is below
// 2^-45 of a.h, which err must cover.
__device__ __forceinline__ void ff_round(ff a, f2 err, float &v0, float &v1, bool &sure0, bool &sure1)
{
    float d0, d1;
    upk2(add2(a.h, add2(a.l, err)), v0, v1);
    upk2(add2(a.h, sub2(a.l, err)), d0, d1);
    sure0 = v0 == d0 && fabsf(v0) >= 0x1p-70f;
    sure1 = v1 == d1 && fabsf(v1) >= 0x1p-70f;
}

}  // namespace pwa
