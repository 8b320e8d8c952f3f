// split_math.cuh -- numbers held as an unevaluated sum of two floats.
//
// A GB300 SM partition issues an FP64 instruction of a warp every 64 cycles and
// an FP32 one every cycle, so a product of two pairs (4 instructions) or a sum
// (8) costs an eighth of the FP64 one it stands for.  A pair carries 46 to 48
// significant bits.  It is used where its value enters a double as a small
// correction (a kick against the velocity, f - 1 against 1), so that its error
// lies below the rounding of that double; the sums themselves stay in FP64.
//
// Error-free transforms: Knuth's two-sum, Dekker's fast two-sum and the product
// with its fused remainder.  The __f*_rn intrinsics keep the compiler from
// contracting them.
#pragma once
#include "device_math.cuh"

namespace glisse {

struct F2 {
    float h, l;
};

// x rounded to a pair (conversions: for constants)
__host__ __device__ inline F2 f2_const(double x) {
    const float h = (float)x;
    return F2{h, (float)(x - (double)h)};
}

__device__ __forceinline__ float rsqrt_f32(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_f32(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// a + b = s + e exactly (6 instructions).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// The same for |a| >= |b| (3 instructions).
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

__device__ __forceinline__ F2 f2_norm(float h, float l) {
    F2 r;
    fast_two_sum(h, l, r.h, r.l);
    return r;
}

// Product; the low part may reach 2^-22 of the high one (not renormalised).
__device__ __forceinline__ F2 f2_mul(const F2& a, const F2& b) {
    F2 r;
    r.h = __fmul_rn(a.h, b.h);
    r.l = __fmaf_rn(a.h, b.h, -r.h);
    r.l = __fmaf_rn(a.h, b.l, r.l);
    r.l = __fmaf_rn(a.l, b.h, r.l);
    return r;
}

__device__ __forceinline__ F2 f2_add(const F2& a, const F2& b) {
    F2 r;
    float e;
    two_sum(a.h, b.h, r.h, e);
    r.l = __fadd_rn(e, __fadd_rn(a.l, b.l));
    return r;
}

__device__ __forceinline__ F2 f2_sub(const F2& a, const F2& b) {
    F2 r;
    float e;
    two_sum(a.h, -b.h, r.h, e);
    r.l = __fadd_rn(e, __fsub_rn(a.l, b.l));
    return r;
}

// Quotient a / b with rb ~ 1 / b.h (2^-22).
__device__ __forceinline__ F2 f2_div(const F2& a, const F2& b, float rb) {
    F2 q;
    q.h = __fmul_rn(a.h, rb);
    float e = __fmaf_rn(-q.h, b.h, a.h);
    e = __fadd_rn(__fmaf_rn(-q.h, b.l, e), a.l);
    q.l = __fmul_rn(e, rb);
    return q;
}

// a - b c
__device__ __forceinline__ F2 f2_fnma(const F2& b, const F2& c, const F2& a) { return f2_sub(a, f2_mul(b, c)); }

// D^(-1/2) of a pair to 46 bits: y, y^2 = yy + yl exactly, e = 1 - D y^2 (below 2^-21).
struct RsqrtF2 {
    float y, yy, yl, e;
};
__device__ __forceinline__ RsqrtF2 f2_rsqrt(const F2& D) {
    RsqrtF2 r;
    r.y = rsqrt_f32(D.h);
    r.yy = __fmul_rn(r.y, r.y);
    r.yl = __fmaf_rn(r.y, r.y, -r.yy);
    r.e = __fmaf_rn(-D.h, r.yy, 1.0f);
    r.e = __fmaf_rn(-D.h, r.yl, r.e);
    r.e = __fmaf_rn(-D.l, r.yy, r.e);
    return r;
}

// k D^(-3/2) = k y^3 (1 - e)^(-3/2), k D^(-1) = k y^2 / (1 - e)
__device__ __forceinline__ F2 f2_k_rcube(const RsqrtF2& r, const F2& k) {
    const float y3 = __fmul_rn(r.y, r.yy);
    const float y3l = __fmaf_rn(r.y, r.yl, __fmaf_rn(r.y, r.yy, -y3));
    F2 s;
    s.h = __fmul_rn(k.h, y3);
    s.l = __fmaf_rn(k.h, y3, -s.h);
    s.l = __fmaf_rn(k.l, y3, s.l);
    s.l = __fmaf_rn(k.h, y3l, s.l);
    s.l = __fmaf_rn(s.h, r.e * __fmaf_rn(1.875f, r.e, 1.5f), s.l);
    return s;
}

// |a|^2 of a split vector
__device__ __forceinline__ F2 f2_norm2(const F2 (&a)[3]) {
    float p[3], q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        p[c] = __fmul_rn(a[c].h, a[c].h);
        q[c] = __fmaf_rn(a[c].h, a[c].h, -p[c]);
        q[c] = __fmaf_rn(__fmaf_rn(2.0f, a[c].h, a[c].l), a[c].l, q[c]);
    }
    F2 r;
    float e0, e1;
    two_sum(p[0], p[1], r.h, e0);
    two_sum(r.h, p[2], r.h, e1);
    r.l = __fadd_rn(__fadd_rn(e0, e1), __fadd_rn(__fadd_rn(q[0], q[1]), q[2]));
    return r;
}

// (a.x b.x + a.y b.y) + a.z b.z from split vectors.
__device__ __forceinline__ F2 f2_dot(const F2 (&a)[3], const F2 (&b)[3]) {
    const F2 p = f2_mul(a[0], b[0]), q = f2_mul(a[1], b[1]), r = f2_mul(a[2], b[2]);
    F2 s;
    float e, f;
    two_sum(p.h, q.h, s.h, e);
    two_sum(s.h, r.h, s.h, f);
    s.l = __fadd_rn(__fadd_rn(e, f), __fadd_rn(__fadd_rn(p.l, q.l), r.l));
    return s;
}

// A double as a pair, by integer operations and one int-to-float conversion
// (an F2F conversion occupies the FP64 pipe): the leading 24 bits, and the other
// 29 rounded to 24.  |x| below 2^-74 is read as 2^-74 (1 + ...): far below
// anything it is added to.  |x| must be below 2^127.
__device__ __forceinline__ F2 f2_split(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned a = max(hi & 0x7FFFFFFFu, (unsigned)(1023 - 74) << 20);
    const unsigned b = (__funnelshift_l(lo, a, 3) + 0x40000000u) | (hi & 0x80000000u);
    F2 r;
    r.h = __uint_as_float(b);
    r.l = __fmul_rn((float)(int)(lo & 0x1FFFFFFFu), __uint_as_float((b & 0xFF800000u) - (52u << 23)));
    return r;
}

// A positive double's leading 24 bits (truncated) as a float; x in the float's normal range.
__device__ __forceinline__ float f32_trunc(double x) {
    return __uint_as_float(__funnelshift_l((unsigned)__double2loint(x), (unsigned)__double2hiint(x), 3) + 0x40000000u);
}

// y^2 exactly for a float y of at most 21 significant bits (in [2^-60, 2^60]).
__device__ __forceinline__ double f21_square(float y) {
    const unsigned b = __float_as_uint(y);
    const unsigned m = ((b & 0x7FFFFFu) | 0x800000u) >> 3;       // y = m 2^(ey - 147)
    const unsigned long long m2 = (unsigned long long)m * m;     // [2^40, 2^42)
    const int a = (int)(m2 >> 41);
    return __longlong_as_double(((long long)(2 * (int)(b >> 23) + 768 + a) << 52) + (long long)(m2 << (12 - a)));
}

// k y^3 correctly rounded (ties away from zero) for a float y > 0 of at most 21 significant
// bits, by integer arithmetic as in seed_square_kcube; its range check is the caller's
// (y in [2^-60, 2^60], k normal).
__device__ __forceinline__ double f21_kcube(float y, double k) {
    const unsigned b = __float_as_uint(y);
    const int ey = (int)(b >> 23);                              // y = m 2^(ey - 147)
    const unsigned m = ((b & 0x7FFFFFu) | 0x800000u) >> 3;     // [2^20, 2^21)
    const unsigned long long m3 = (unsigned long long)m * m * m;  // [2^60, 2^63)
    const long long kb = __double_as_longlong(k);
    const int ek = (int)((kb >> 52) & 0x7FF);
    const unsigned long long km = ((unsigned long long)kb & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const unsigned long long p = __umul64hi(km << 11, m3 << 1);
    const int sh = 11 - __clzll(p);
    const unsigned long long q = ((p >> (sh - 1)) + 1) >> 1;
    const int be = sh + ek + 3 * (ey + 896) - 3077;
    return __longlong_as_double((((long long)(be - 1) << 52) + (long long)q) | (kb & (long long)(1ull << 63)));
}

// A normalised pair (|l| <= ulp(h)) as a double: h's bits moved to a double,
// then l added to the significand as an integer in units of 2^-46 of h's binade
// (l beyond them is dropped: below 2^-47 of the value).  Below a power of two
// the significand's unit is half as large, so a negative l counts double there.
// Pairs below 2^-80 lose their l.
__device__ __forceinline__ double f2_double(const F2& v) {
    const unsigned b = __float_as_uint(v.h);
    const unsigned hw = ((unsigned)((int)b >> 3) & 0x8FFFFFFFu) + 0x38000000u;
    const long long base = ((long long)hw << 32) | (b << 29);
    // sign(h) 2^(46 - E): k = l / h's binade in units of 2^-46, toward h's sign
    const float sc = __uint_as_float(((b ^ 0x7F800000u) & 0xFF800000u) + (45u << 23));
    const float magic = 12582912.0f;  // 1.5 2^23
    int k = (int)__float_as_uint(__fmaf_rn(v.l, sc, magic)) - 0x4B400000;
    if (k < 0 && (b & 0x007FFFFFu) == 0u) k += k;
    return __longlong_as_double(base + (long long)k * 64);
}

}  // namespace glisse
