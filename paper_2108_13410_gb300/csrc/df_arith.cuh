// df_arith.cuh -- double-float arithmetic on packed FP32x2 registers, (re, im) of the high
// and of the low parts in one 64-bit register each (xpass_df.cuh says what it is for).
#pragma once
#include "packed.cuh"

namespace qsim {

__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 swap2(u64 a) {   // (x, y) -> (y, x)
    u64 d;
    asm("{\n\t.reg .b32 x, y;\n\tmov.b64 {x, y}, %1;\n\tmov.b64 %0, {y, x};\n\t}" : "=l"(d) : "l"(a));
    return d;
}

// a * b - p per lane for p = RN(a * b): exact, by scalar FMA
__device__ __forceinline__ u64 prod_err(u64 a, u64 b, u64 p) {
    const float2 x = unpk(a), y = unpk(b), q = unpk(p);
    return pk(fmaf(x.x, y.x, -q.x), fmaf(x.y, y.y, -q.y));
}

// (vh, vl) * (ch, cl), both lanes: exact high product, cross terms, renormalisation.
__device__ __forceinline__ void df_mul(u64 vh, u64 vl, u64 ch, u64 cl, u64 &rh, u64 &rl) {
    const u64 p = mul2(vh, ch);
    u64 e = prod_err(vh, ch, p);
    e = fma2p(vh, cl, e);
    e = fma2p(vl, ch, e);
    rh = add2(p, e);
    rl = sub2(e, sub2(rh, p));
}

__device__ __forceinline__ void df_add(u64 ah, u64 al, u64 bh, u64 bl, u64 &rh, u64 &rl) {
    const u64 s = add2(ah, bh);
    const u64 sv = sub2(s, ah);
    u64 e = add2(sub2(ah, sub2(s, sv)), sub2(bh, sv));
    e = add2(e, add2(al, bl));
    rh = add2(s, e);
    rl = sub2(e, sub2(rh, s));
}

// sum and difference without renormalisation (see the header)
__device__ __forceinline__ void df_butterfly_lazy(u64 &ah, u64 &al, u64 &bh, u64 &bl) {
    const u64 s = add2(ah, bh);
    const u64 sv = sub2(s, ah);
    const u64 es = add2(sub2(ah, sub2(s, sv)), sub2(bh, sv));
    const u64 d = sub2(ah, bh);
    const u64 dv = sub2(d, ah);
    const u64 ed = sub2(sub2(ah, sub2(d, dv)), add2(bh, dv));
    const u64 ls = add2(es, add2(al, bl));
    const u64 ld = add2(ed, sub2(al, bl));
    ah = s; al = ls; bh = d; bl = ld;
}

// t * x for a double-float scalar t = (th, th) + (tl, tl) and pair x: unnormalised
// product (p, e), p = RN(th xh), e = its exact error plus the cross terms
__device__ __forceinline__ void df_scale_lazy(u64 th, u64 tl, u64 xh, u64 xl, u64 &p, u64 &e) {
    p = mul2(th, xh);
    e = prod_err(th, xh, p);
    e = fma2p(th, xl, e);
    e = fma2p(tl, xh, e);
}

// tangent-form rotation of a pair, without renormalisation: a' = a + t b, b' = b - t a
__device__ __forceinline__ void df_rot_lazy(u64 &ah, u64 &al, u64 &bh, u64 &bl, u64 th, u64 tl) {
    u64 pb, eb, pa, ea;
    df_scale_lazy(th, tl, bh, bl, pb, eb);
    df_scale_lazy(th, tl, ah, al, pa, ea);
    const u64 s = add2(ah, pb);
    const u64 sv = sub2(s, ah);
    const u64 es = add2(sub2(ah, sub2(s, sv)), sub2(pb, sv));
    const u64 ls = add2(es, add2(al, eb));
    const u64 d = sub2(bh, pa);
    const u64 dv = sub2(d, bh);
    const u64 ed = sub2(sub2(bh, sub2(d, dv)), add2(pa, dv));
    const u64 ld = add2(ed, sub2(bl, ea));
    ah = s; al = ls; bh = d; bl = ld;
}

// v * i^k on both parts (exact)
__device__ __forceinline__ void df_ipow(u64 &h, u64 &l, int k) {
    const float2 a = mul_ipow(unpk(h), k), b = mul_ipow(unpk(l), k);
    h = pk(a.x, a.y);
    l = pk(b.x, b.y);
}

// Phase table entry in double-float, packed for the complex product
// v (c + i s) = (vr c - vi s, vi c + vr s) = v*(c, c) + swap(v*(s, -s)).
struct DfPhase { u64 ch, cl, sh, sl; };

__device__ __forceinline__ void df_phase(u64 &vh, u64 &vl, const DfPhase &q) {
    u64 ah, al, bh, bl;
    df_mul(vh, vl, q.ch, q.cl, ah, al);   // (vr c, vi c)
    df_mul(vh, vl, q.sh, q.sl, bh, bl);   // (vr s, -vi s)
    df_add(ah, al, swap2(bh), swap2(bl), vh, vl);
}

// Split of a double into two floats with integer operations (GB300's FP64 conversions
// run at the FP64 rate): hi = d with its binary fraction cut to 23 bits (truncation),
// lo = the 29 dropped fraction bits as a float (rounded to 24 bits), so hi + lo keeps 48
// significand bits.  |d| below 2^-126 (no normal float hi) maps to (0, 0): the state's
// amplitudes are at most 1, so that drops less than 2^-126 absolute.
__device__ __forceinline__ void split_double(double d, float &hi, float &lo) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(d);
    const unsigned int top = (unsigned int)(u >> 32), bot = (unsigned int)u;
    const unsigned int sign = top & 0x80000000u;
    const int e = (int)((top >> 20) & 0x7ffu);          // biased double exponent
    const int E = e - 896;                               // biased float exponent of hi
    if (e == 0x7ff || E >= 255) { hi = __double2float_rn(d); lo = 0.f; return; }   // keeps inf / NaN
    if (E <= 0) { hi = 0.f; lo = 0.f; return; }
    hi = __uint_as_float(sign | ((unsigned int)E << 23) | ((top & 0xfffffu) << 3) | (bot >> 29));
    const unsigned int r = bot & 0x1fffffffu;            // dropped bits, units of 2^(e-1075)
    const int El = e - 948;                              // biased float exponent of 2^(e-1075)
    // below the normal range the power of two is applied in two factors (El + 64 > 12 here)
    const float v = El > 0 ? __uint2float_rn(r) * __uint_as_float((unsigned int)El << 23)
                           : __uint2float_rn(r) * __uint_as_float((unsigned int)(El + 64) << 23) * 0x1p-64f;
    lo = __uint_as_float(__float_as_uint(v) | sign);
}

// hi + lo as a double: exact conversions of both floats by bit assembly, one FP64 add
__device__ __forceinline__ double float_to_double_bits(float f) {
    const unsigned int b = __float_as_uint(f);
    const unsigned int E = (b >> 23) & 0xffu;
    if (E == 0 || E == 255) return (double)f;            // zero, subnormal, inf, NaN
    const unsigned long long d = ((unsigned long long)(b & 0x80000000u) << 32) |
                                 ((unsigned long long)(E + 896u) << 52) |
                                 ((unsigned long long)(b & 0x7fffffu) << 29);
    return __longlong_as_double((long long)d);
}

// (re, im) of a pair as complex128
__device__ __forceinline__ double2 df_join(u64 vh, u64 vl) {
    const float2 h = unpk(vh), l = unpk(vl);
    return make_double2(float_to_double_bits(h.x) + float_to_double_bits(l.x),
                        float_to_double_bits(h.y) + float_to_double_bits(l.y));
}

}  // namespace qsim
