// split_step.cuh -- the particle's drift and kick with FP64 where a result is
// formed and float pairs (split_math.cuh) for the corrections to it.
//
// Of a step's position, velocity and their increments only the sums need 53
// bits: a kick is 1e-3 of the velocity or less and f - 1, gdot - 1 and dt - g are
// (n dt)^2 or less, so 46 bits of them reach below the last bit of the sum.
// One step then takes 19 FP64 instructions (r^2 and dt mu / r^3: 5; g, fdot: 2;
// f x + g v: 6; fdot x: 3; gdot v and the kick, summed in pairs: 3) against 61 + 12 N_p for
// the all-FP64 step, and ~1200 instructions in all, which fit under them.
// Measured (1048576 particles, 4 planets, 1024 steps): 44.8 ms against 207 ms; the 19
// instructions at 65 cycles are 73% of that.  Against 113-bit arithmetic, one step's velocity
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
// other lanes.
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
// The drift for longer steps (m or b above kSplitZ, up to kWideZ: a planet-crossing
// particle near its pericentre, a short-period system).  The corrections reach
// 2^-4 there, so the pairs are kept to 2^-48 of their own values: products are
// normalised (f2_muln), k, e2 = 2 g2 - 1 and 1/D - 1 are summed from small values
// and never through a number near 1, S is a pair, and f - 1 starts from m in FP64:
//   f - 1 = -(m/2) (1 + e2),  gdot - 1 = (f - 1) (1 + kd),  kd = 1/D - 1.
// ~700 instructions and 2 FP64 ones more than drift_split, against ~63 FP64 ones for
// the all-FP64 drift.  Its error is the FP64 drift's up to b = 0.015 (v 0.74 against
// 0.65 units of 2^-53) and 0.99 against 0.67 at 0.03, where the kick's fewer roundings
// still keep the step below the all-FP64 one; beyond, the FP64 drift.
// ---------------------------------------------------------------------------
constexpr float kWideZ = 0.046875f;  // 3/64
constexpr float kWideA = 0.0625f;    // 2^-4

// c + x y for |c| above |x y| (c: a constant's pair)
__device__ __forceinline__ F2 f2_horner(const F2& c, const F2& x, const F2& y) {
    const F2 p = f2_mul(x, y);
    F2 r;
    float e;
    fast_two_sum(c.h, p.h, r.h, e);
    r.l = __fadd_rn(__fadd_rn(e, c.l), p.l);
    return r;
}

__device__ __forceinline__ bool drift_wide(double r2, double mudt, double dt, const F2& dt2, const double (&s)[6],
                                           DriftFactors& out) {
    F2 u, v2;
    {
        const F2 x[3] = {f2_split_near(s[0]), f2_split_near(s[1]), f2_split_near(s[2])};
        const F2 v[3] = {f2_split_near(s[3]), f2_split_near(s[4]), f2_split_near(s[5])};
        u = f2_dotn(x, v);
        v2 = f2_dotn(v, v);
    }
    F2 w;
    double dts;
    inverse_powers(r2, mudt, w, dts);
    const F2 dw = f2_muln(dt2, w);
    const F2 a = f2_muln(u, dw);
    const F2 n = f2_muln(v2, f2_muln(dt2, dw));
    const double md = dt * dts;
    const F2 m = f2_split(md);
    const F2 q = f2_sub(n, m);
    const F2 b = f2_sub(m, q);

    // ---- S in FP32 ----
    float S = __fmaf_rn(-1.0f / 6.0f, q.h, __fmaf_rn(0.5f * a.h, a.h - 1.0f, 1.0f));
#pragma unroll
    for (int it = 0; it < 3; ++it) {
        const float s2 = S * S, z = b.h * s2;
        const float g2 = s2 * __fmaf_rn(z, __fmaf_rn(z, __fmaf_rn(z, -1.0f / 40320.0f, 1.0f / 720.0f), -1.0f / 24.0f),
                                        0.5f);
        const float g3 = s2 * S * __fmaf_rn(z, __fmaf_rn(z, 1.0f / 5040.0f, -1.0f / 120.0f), 1.0f / 6.0f);
        const float F = __fmaf_rn(a.h, g2, __fmaf_rn(q.h, g3, S - 1.0f));
        const float D = __fmaf_rn(q.h, g2, __fmaf_rn(a.h, 1.0f - __fmaf_rn(a.h, g2, m.h * g3), 1.0f));
        S = __fmaf_rn(-F, rcp_f32(D), S);
    }
    // ---- at S: 2 g2 = (1 + sm)(1 + t2) = 1 + e2,  6 g3 = S^3 (1 + t3) ----
    F2 s2, s3;
    s2.h = __fmul_rn(S, S);
    s2.l = __fmaf_rn(S, S, -s2.h);
    s3.h = __fmul_rn(s2.h, S);
    s3.l = __fmaf_rn(s2.l, S, __fmaf_rn(s2.h, S, -s3.h));
    const F2 z = f2_muln(b, s2);
    const float zh = z.h;
    // t2 = z (-1/12 + z/360 - z^2/20160 + z^3/1814400 - ...), t3 = z (-1/20 + z/840 - z^2/60480 + ...)
    constexpr F2 p21 = {-0.083333336f, 2.483527e-09f}, p22 = {0.0027777778f, -6.726219e-11f},
                 p23 = {-4.9603175e-05f, 6.813992e-13f};
    constexpr F2 p31 = {-0.05f, 7.4505807e-10f}, p32 = {0.0011904762f, -4.5457412e-11f};
    F2 t2, t3;
    {
        const float y2 = zh * __fmaf_rn(zh, __fmaf_rn(zh, 2.294149e-11f, -4.175351e-09f), 5.511464e-07f);
        F2 h2;
        fast_two_sum(p23.h, y2, h2.h, h2.l);
        h2.l = __fadd_rn(h2.l, p23.l);
        t2 = f2_muln(z, f2_horner(p21, z, f2_horner(p22, z, h2)));
        const float y3 = zh * __fmaf_rn(zh, __fmaf_rn(zh, -9.635426e-10f, 1.5031264e-07f), -1.6534392e-05f);
        F2 h3;
        fast_two_sum(p32.h, y3, h3.h, h3.l);
        h3.l = __fadd_rn(h3.l, p32.l);
        t3 = f2_muln(z, f2_horner(p31, z, h3));
    }
    const F2 sm = f2_norm(__fsub_rn(s2.h, 1.0f), s2.l);
    F2 e2 = f2_add(f2_add(sm, t2), f2_mul(sm, t2));
    F2 g3 = f2_mul(s3, t3);  // 6 g3 = s3 + s3 t3
    {
        float t;
        fast_two_sum(s3.h, g3.h, g3.h, t);
        g3.l = __fadd_rn(t, __fadd_rn(s3.l, g3.l));
    }
    const F2 a2 = {0.5f * a.h, 0.5f * a.l}, q2 = {0.5f * q.h, 0.5f * q.l};
    constexpr F2 k6 = {0.16666667f, -4.967054e-09f};
    const F2 q6 = f2_muln(q, k6), m6 = f2_muln(m, k6);
    const F2 ag = f2_add(a2, f2_mul(a2, e2));   // a g2
    const F2 qg = f2_add(q2, f2_mul(q2, e2));   // q g2
    const F2 q3 = f2_mul(q6, g3), m3 = f2_mul(m6, g3);  // q g3, m g3
    const F2 S1 = {__fsub_rn(S, 1.0f), 0.0f};
    // F = (S - 1) + a g2 + q g3; y1 = g1 - 1 = (S - 1) - b g3; rho = D - 1 = a + a y1 + q g2
    const F2 F = f2_normp(f2_add(f2_add(S1, ag), q3));
    const F2 y1 = f2_add(f2_sub(S1, m3), q3);
    F2 rho = f2_add(f2_add(a, f2_mul(a, y1)), qg);
    // d = -F / D as a pair
    const float rD0 = rcp_f32(__fadd_rn(1.0f, rho.h));
    F2 d;
    d.h = __fmul_rn(-F.h, rD0);
    // residual F + d D = (F.h + d.h) + F.l + d.h rho
    d.l = __fmul_rn(__fadd_rn(__fadd_rn(F.h, d.h), __fmaf_rn(d.h, rho.h, F.l)), -rD0);
    const bool ok = fabsf(a.h) <= kWideA && fabsf(b.h) <= kWideZ && m.h <= kWideZ && fabsf(d.h) <= 3.8146973e-6f;
    // to S + d (second order in d included): g2 + d g1 + d^2 g0 / 2, g3 + d g2, y1 + d g0, D + d (a g0 + q g1)
    const float g0f = __fmaf_rn(-b.h, __fmaf_rn(0.5f, e2.h, 0.5f), 1.0f), g1f = __fadd_rn(1.0f, y1.h);
    const float dy = __fmaf_rn(0.5f * d.h, g0f, y1.h);  // g1 - 1 halfway
    const F2 dg2 = f2_norm(d.h, __fmaf_rn(d.h, dy, d.l));  // g2(S + d) - g2
    e2 = f2_add(e2, F2{2.0f * dg2.h, 2.0f * dg2.l});
    const float dg3 = d.h * __fmaf_rn(0.5f * d.h, g1f, __fmaf_rn(0.5f, e2.h, 0.5f));
    const F2 mg3 = f2_add(m3, F2{m.h * dg3, 0.0f});
    const F2 T = f2_add(f2_add(a2, f2_mul(a2, e2)), mg3);  // a g2 + m g3 = 1 - g1
    rho = f2_normp(f2_add(f2_sub(a, f2_mul(a, T)), f2_add(q2, f2_mul(q2, e2))));
    F2 N = f2_add(T, rho);
    N = f2_norm(-N.h, -N.l);  // g1 - D
    F2 D;
    fast_two_sum(1.0f, rho.h, D.h, D.l);
    D.l = __fadd_rn(D.l, rho.l);
    const float rD = rcp_f32(D.h);
    const F2 k = f2_divn(N, D, rD), kd = f2_divn(F2{-rho.h, -rho.l}, D, rD);
    const double mh = -0.5 * md;
    out.fm1 = fma(mh, f2_double(f2_normp(e2)), mh);
    F2 e1, kd1;  // 1 + e2, 1 + kd
    fast_two_sum(1.0f, e2.h, e1.h, e1.l);
    e1.l = __fadd_rn(e1.l, e2.l);
    fast_two_sum(1.0f, kd.h, kd1.h, kd1.l);
    kd1.l = __fadd_rn(kd1.l, kd.l);
    out.gdm1 = f2_muln(f2_muln(F2{-0.5f * m.h, -0.5f * m.l}, f2_normp(e1)), f2_normp(kd1));
    out.g = fma(-dt, f2_double(f2_normp(mg3)), dt);
    out.fd = fma(-dts, f2_double(k), -dts);
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
