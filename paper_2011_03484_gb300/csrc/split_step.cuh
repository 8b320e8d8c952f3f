// split_step.cuh -- the particle's drift and kick with FP64 where a result is
// formed and float pairs (split_math.cuh) for the corrections to it.
//
// Of a step's position, velocity and their increments only the sums need 53
// bits: a kick is 1e-3 of the velocity or less and f - 1, gdot - 1 and dt - g are
// (n dt)^2 or less, so 46 bits of them reach below the last bit of the sum.
// One step then takes 19 FP64 instructions (r^2 and dt mu / r^3: 5; g, fdot: 2;
// f x + g v: 6; fdot x: 3; gdot v and the kick, summed in pairs: 3) against 61 + 12 N_p for
// the all-FP64 step, and ~1200 instructions in all, which fit under them.
// Measured (1048576 particles, 4 planets, 1024 steps): 46.4 ms against 207 ms; the 19
// instructions at 65 cycles are 71% of that.  Against 113-bit arithmetic, one step's velocity
// is off by 0.58 to 0.71 units of 2^-53 (rms over belts of 20-100 AU; the all-FP64 step:
// 1.09 to 1.21): fewer roundings, and what the pairs drop lies below them.
#pragma once
#include "glisse_internal.h"
#include "split_math.cuh"

namespace glisse {

// The particle constants as the pairs this file works with.
struct SplitConsts {
    F2 dt;
    double mudt;             // mu dt
    F2 tg[kMaxPlanets];      // dt G m_j
    float rc2[kMaxPlanets];  // R_crit,j^2, rounded up by more than a float's error
};

__host__ __device__ inline void split_planet(const ParticleConsts& pc, int j, SplitConsts& sc) {
    sc.tg[j] = f2_const(pc.tgm_full[j]);
    sc.rc2[j] = (float)(pc.rc2[j] * (1.0 + 0x1p-20));
}

__host__ __device__ inline void split_step_consts(const ParticleConsts& pc, SplitConsts& sc) {
    sc.dt = f2_const(pc.dt);
    sc.mudt = pc.mu * pc.dt;
}

// ---------------------------------------------------------------------------
// Drift.  With h = dt / r0 and S = s r0 / dt the universal variable, the time
// equation and r / r0 become
//   g1 + a g2 + m g3 = 1,   D = r / r0 = 1 + a g1 + q g2,
//   a = dt (r.v) / r0^2,  m = mu dt^2 / r0^3,  n = dt^2 v^2 / r0^2,
//   q = n - m,  b = m - q (= beta h^2),  g_k = S^k c_k(b S^2),  g1 = 1 - a g2 - m g3
// (r0 G_0 + ... with G_k = (dt/r0)^k g_k).  All are small but S, g1, D ~ 1, and
//   f - 1 = -m g2,  g = dt - dt m g3,  gdot - 1 = -m g2 / D,
//   fdot = -(dt mu / r0^3) g1 / D = -(dt mu / r0^3) (1 + k)
// so the factors of x and v come from pairs except for dt and dt mu / r0^3, which
// are FP64.  S: series start, one Newton step in FP32, one in pairs (the error
// left is below (a/2) (2^-18)^2).
// Domain: |a| <= kSplitA, b and m <= kSplitZ; the caller runs the FP64 drift for
// other lanes.  (A form of the pairs kept to 2^-48 for steps up to m = 3/64 took 7700 cycles for
// a lone warp against the FP64 drift's 4500, and 15% more on orbits up to e = 0.9.)
// ---------------------------------------------------------------------------
constexpr float kSplitZ = 0.00390625f;  // 2^-8
constexpr float kSplitA = 0.046875f;    // 3/64

// |x| and |v| of a particle whose r^2 has this exponent are well inside the floats' range.
__device__ __forceinline__ bool in_float_range(double r2) { return (unsigned)(exp_bits(r2) - (1023 - 100)) <= 200u; }

// |v|^2 and |v|^2 / |r|^2 to a float's precision; v2 negative outside the floats' range.
struct Speed {
    float v2, rate2;
};

__device__ __forceinline__ Speed float_speed(double r2, double vx, double vy, double vz) {
    const float a = d2f_bits(vx), b = d2f_bits(vy), c = d2f_bits(vz);
    const float v2 = fmaf(a, a, fmaf(b, b, c * c));
    return Speed{in_float_range(r2) ? v2 : -1.0f, __fdividef(v2, d2f_bits(r2))};
}

// True where m = mu dt^2 / r^3 alone puts a lane outside drift_split's domain.
__device__ __forceinline__ bool beyond_split(double r2, float mudt, float dt) {
    const float y = rsqrt_f32(f32_trunc(r2));
    return in_float_range(r2) && mudt * dt * (y * y * y) > 1.001f * kSplitZ;
}

struct DriftFactors {
    double fm1, g, fd;
    F2 gdm1;
};

// Scalars of drift_split for the derivatives of the drift (split_diff.cuh): those of its
// comment, S = S + d, T = 1 - g1, rho = D - 1, rD ~ 1/D, k = (g1 - D) / D, w = 1 / r0^2 (wd: in FP64),
// dts = dt mu / r0^3 (dts2: as a pair), fm1 = f - 1.
struct DriftSeries {
    F2 a, m, q, b, w, dts2, g2, g3, T, rho, D, k, fm1;
    float rD, S, d;
    double dts, wd;
};

// w = 1 / r0^2 as a pair (and, into wd, as a double) and dts = dt mu / r0^3 (mudt = mu dt) from r0^2.
__device__ __forceinline__ void inverse_powers(double r2, double mudt, F2& w, double& dts, double* wd = nullptr) {
    // y ~ 1 / r0 (21 bits), e = 1 - r0^2 y^2;
    // dt mu / r0^3 = dt mu y^3 (1 - e)^(-3/2) = dt mu y^3 (1 + 3e/2 + 15e^2/8 + ...)
    const float y = __uint_as_float(__float_as_uint(rsqrt_f32(f32_trunc(r2))) & 0xFFFFFFF8u);
    const double y2 = f21_square(y);
    const F2 er = f2_split(fma(-r2, y2, 1.0));
    F2 c;
    c.h = __fmul_rn(1.5f, er.h);
    c.l = __fmaf_rn(1.5f, er.l, __fmaf_rn(1.875f * er.h, er.h, __fmaf_rn(1.5f, er.h, -c.h)));
    const double dt3 = f21_kcube(y, mudt);
    dts = fma(dt3, f2_double(f2_norm(c.h, c.l)), dt3);
    // 1 / r0^2 = y^2 / (1 - e)
    if (wd) *wd = fma(y2, f2_double(f2_norm(er.h, __fmaf_rn(er.h, er.h, er.l))), y2);
    const float yy = __fmul_rn(y, y), yl = __fmaf_rn(y, y, -yy), p = __fmul_rn(yy, er.h);
    float e;
    fast_two_sum(yy, p, w.h, e);
    w.l = __fadd_rn(__fadd_rn(e, __fmaf_rn(yy, er.h, -p)),
                    __fmaf_rn(yy, __fmaf_rn(er.h, er.h, er.l), __fmaf_rn(yl, er.h, yl)));
}

// drift_split's speed alone.
__device__ __forceinline__ Speed split_speed(double r2, double mudt, const F2 (&v)[3]) {
    F2 w;
    double dts;
    inverse_powers(r2, mudt, w, dts);
    const F2 v2 = f2_dot(v, v);
    return Speed{v2.h, v2.h * w.h};
}

// mudt = mu dt, dt2 = dt; ser (or null) receives the scalars.
__device__ __forceinline__ bool drift_split(double r2, double mudt, double dt, const F2& dt2, const F2 (&x)[3],
                                            const F2 (&v)[3], DriftFactors& out, Speed& sp,
                                            DriftSeries* ser = nullptr) {
    const F2 u = f2_dot(x, v), v2 = f2_dot(v, v);
    F2 w;
    double dts;
    inverse_powers(r2, mudt, w, dts, ser ? &ser->wd : nullptr);
    const F2 dw = f2_mul(dt2, w);
    const F2 a = f2_mul(u, dw);
    const F2 n = f2_mul(v2, f2_mul(dt2, dw));
    sp = Speed{v2.h, v2.h * w.h};
    const F2 dts2 = f2_split(dts);
    const F2 m = f2_mul(dt2, dts2);
    const F2 q = f2_sub(n, m);
    const F2 b = f2_sub(m, q);

    // ---- S in FP32: S + a S^2 / 2 + q S^3 / 6 + ... = 1 ----
    float S = __fmaf_rn(-1.0f / 6.0f, q.h, __fmaf_rn(0.5f * a.h, a.h - 1.0f, 1.0f));
    {
        const float s2 = S * S, z = b.h * s2;
        const float g2 = s2 * __fmaf_rn(z, __fmaf_rn(z, 1.0f / 720.0f, -1.0f / 24.0f), 0.5f);
        const float g3 = s2 * S * __fmaf_rn(z, -1.0f / 120.0f, 1.0f / 6.0f);
        const float F = __fmaf_rn(a.h, g2, __fmaf_rn(q.h, g3, S - 1.0f));
        const float D = __fmaf_rn(q.h, g2, __fmaf_rn(a.h, 1.0f - __fmaf_rn(a.h, g2, m.h * g3), 1.0f));
        S = __fmaf_rn(-F, rcp_f32(D), S);
    }
    // ---- c2, c3, g2, g3 at S ----
    F2 s2, s3;
    s2.h = __fmul_rn(S, S);
    s2.l = __fmaf_rn(S, S, -s2.h);
    s3.h = __fmul_rn(s2.h, S);
    s3.l = __fmaf_rn(s2.l, S, __fmaf_rn(s2.h, S, -s3.h));
    const F2 z = f2_mul(b, s2);
    const float zz = z.h * z.h;
    constexpr F2 k24 = {-0.0416666679f, 1.24176334e-9f};    // -1/24
    constexpr F2 k120 = {-0.00833333377f, 4.34617164e-10f};  // -1/120
    constexpr F2 k6 = {0.16666667f, -4.96705355e-9f};        // 1/6
    // z c2' with c2' = -1/24 + z / 720 - ... in pairs
    const float p720 = z.h * __fmaf_rn(z.h, -1.0f / 40320.0f, 1.0f / 720.0f);
    F2 c2;
    fast_two_sum(k24.h, p720, c2.h, c2.l);
    c2.l = __fadd_rn(c2.l, k24.l);
    c2 = f2_mul(z, c2);
    F2 c3 = f2_mul(z, k120);
    c3.l = __fmaf_rn(zz, __fmaf_rn(z.h, -1.0f / 362880.0f, 1.0f / 5040.0f), c3.l);
    {
        float t;
        fast_two_sum(0.5f, c2.h, c2.h, t);
        c2.l = __fadd_rn(t, c2.l);
        fast_two_sum(k6.h, c3.h, c3.h, t);
        c3.l = __fadd_rn(t, __fadd_rn(c3.l, k6.l));
    }
    F2 g2 = f2_mul(s2, c2), g3 = f2_mul(s3, c3);
    // ---- Newton step in pairs: F = (S - 1) + a g2 + q g3 ----
    F2 ag2 = f2_mul(a, g2);
    const F2 qg3 = f2_mul(q, g3);
    float F, t;
    two_sum(__fsub_rn(S, 1.0f), ag2.h, F, t);
    F = __fadd_rn(__fadd_rn(F, qg3.h), __fadd_rn(t, __fadd_rn(ag2.l, qg3.l)));
    const float g1f = 1.0f - __fmaf_rn(m.h, g3.h, ag2.h);
    const float Df = __fmaf_rn(q.h, g2.h, __fmaf_rn(a.h, g1f, 1.0f));
    const float d = -F * rcp_f32(Df);
    const bool ok = fabsf(a.h) <= kSplitA && fabsf(b.h) <= kSplitZ && m.h <= kSplitZ && fabsf(d) <= 3.8146973e-6f;
    // g2(S + d) = g2 + d (g1 + d/2), g3(S + d) = g3 + d (g2 + d/2 g1)
    const float d1 = d * __fmaf_rn(0.5f, d, g1f);
    g2.l = __fadd_rn(g2.l, d1);
    g3.l = __fmaf_rn(d, __fmaf_rn(0.5f, d, g2.h), g3.l);
    ag2.l = __fmaf_rn(a.h, d1, ag2.l);
    const F2 mg3 = f2_mul(m, g3);
    // T = 1 - g1 = a g2 + m g3, rho = D - 1 = a g1 + q g2; k = (g1 - D) / D = -(T + rho) / D, summed
    // from the small values (through g1 and D, whose low parts stop at 2^-49, the velocity's
    // error at b = 2^-8 was 1.25 instead of 0.99 units)
    const F2 T = f2_add(ag2, mg3);
    F2 g1, D;
    fast_two_sum(1.0f, -T.h, g1.h, g1.l);
    g1.l = __fsub_rn(g1.l, T.l);
    const F2 rho = f2_add(f2_mul(a, g1), f2_mul(q, g2));
    fast_two_sum(1.0f, rho.h, D.h, D.l);
    D.l = __fadd_rn(D.l, rho.l);
    const float rD = rcp_f32(D.h);
    const F2 N = f2_add(T, rho);
    const F2 k = f2_div(f2_norm(-N.h, -N.l), D, rD);
    F2 mg2 = f2_mul(m, g2);
    mg2 = f2_norm(-mg2.h, -mg2.l);
    const F2 gd = f2_div(mg2, D, rD);
    if (ser) {
        const double wd = ser->wd;
        *ser = DriftSeries{a, m, q, b, w, dts2, g2, g3, T, rho, D, k, mg2, rD, S, d, dts, wd};
    }
    out.fm1 = f2_double(mg2);
    out.gdm1 = gd;
    out.g = fma(-dt, f2_double(f2_norm(mg3.h, mg3.l)), dt);
    out.fd = fma(-dts, f2_double(f2_norm(k.h, k.l)), -dts);
    return ok;
}

// ---------------------------------------------------------------------------
// Kick.  One planet's share s d, s = dt G m / |d|^3, d = r - r_j, added to the sum acc
// with the opposite sign.  P: the planet's position (pairs x, y, z), tg = dt G m.
// Returns false, adding nothing, when the planet is so close that the pairs' error of
// the position (2^-48 |r|) would show in the velocity: s above 0.001 of the orbit's
// angular rate |v| / |r| (lim2: the square), or the encounter radius (squared: rc2,
// rounded up) is near; the caller then forms this term, and the encounter test, in
// FP64.  At 0.01 the largest error of a step's velocity was 36 units of 2^-53 against
// the all-FP64 step's 4.5 (planet-crossing belt), at 0.001 it is 3.6.
// ---------------------------------------------------------------------------
constexpr float kSplitNear2 = 2.0e-6f;              // (0.0014)^2
constexpr float kSplitKick2 = 1.0f / 16384.0f;      // (2^-7)^2

__device__ __forceinline__ bool kick_split(const F2 (&x)[3], const F2 (&P)[3], const F2& tg, float rc2, float lim2,
                                           F2 (&acc)[3]) {
    F2 d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = f2_sub(x[c], P[c]);
    const F2 D = f2_norm2(d);
    F2 s = f2_k_rcube(f2_rsqrt(D), tg);
    const bool far = (s.h * s.h <= lim2) && (D.h >= rc2);
    s.h = far ? s.h : 0.0f;
    s.l = far ? s.l : 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float a = __fmul_rn(-s.h, d[c].h);
        float b = __fmaf_rn(-s.h, d[c].h, -a);
        b = __fmaf_rn(-s.h, d[c].l, b);
        b = __fmaf_rn(-s.l, d[c].h, b);
        float t;
        two_sum(acc[c].h, a, acc[c].h, t);
        acc[c].l = __fadd_rn(acc[c].l, __fadd_rn(t, b));
    }
    return far;
}

}  // namespace glisse
