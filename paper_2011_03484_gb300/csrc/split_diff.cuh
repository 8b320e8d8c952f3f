// split_diff.cuh -- the drift's tangent and adjoint, and the kick's tidal matrix, with
// FP64 sums and float-pair corrections (split_math.cuh).
//
// In the units of drift_split (h = dt / r0, g_k = G_k / h^k) the drift's factors depend on
//   alpha = r.dr / r0^2,  eta = dt (dr.v + r.dv) / r0^2,  kappa = dt^2 v.dv / r0^2:
//   dS = -(g1 alpha + g2 eta + Tb omega) / D,  omega = dbeta h^2 = -2 zeta,  zeta = m alpha + kappa,
//   dg0 = -b g1 dS + gb0 omega,  dg_n = g_(n-1) dS + gb_n omega,  gb_n = -(S g_(n+1) - n g_(n+2)) / 2,
//   Tb = gb1 + a gb2 + m gb3,  theta = dD = alpha g0 + dg0 + eta g1 + a dg1 + m dg2,
//   df = m (g2 alpha - dg2),  dg = -dt m dg3,  dgdot = (m / D)(-dg2 + g2 theta / D),
//   dfdot = (m / dt)(-dg1 / D + (g1 / D)(theta / D + alpha)).
// A state's derivative then changes in a step by dt dv, by fdot dr and by the tide
// 3 (dt mu / r0^5)(r.dr) r, which are of first order in n dt and stay FP64, and by
// corrections of second order, (n dt)^2 <= 2^-8, in pairs.  dfdot's factor of alpha is
// (m / dt)(3 + X) with
//   p = g1 / D = 1 + k,  j = g0 / D - 1,  X = 3 k + p (y + j),  y = j - (1 + j) a p - q p^2,
// so that X, too, is summed from small values.  ~30 FP64 instructions per drift (tangent or
// adjoint) against 119 and 140 for the FP64 form (drift_diff.cuh), which serves the
// lanes outside drift_split's domain.
//
// Cotangents and tangents have any scale: their components enter the pairs divided by
// the power of two of the largest one.
#pragma once
#include "split_step.cuh"

namespace glisse {

// Binary exponent of the largest component; 0 if all are zero.  Returns false beyond
// 2^+-900 (a subnormal, an infinity or a NaN): the FP64 form then.
__device__ __forceinline__ bool scale_exponent(const double (&l)[6], int& e) {
    unsigned h = 0, any = 0;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const unsigned a = (unsigned)__double2hiint(l[c]) & 0x7FFFFFFFu;
        h = max(h, a);
        any |= a | (unsigned)__double2loint(l[c]);
    }
    e = any == 0u ? 0 : (int)(h >> 20) - 1023;
    return (unsigned)(e + 900) <= 1800u;
}

// x 2^-e as a pair, |x 2^-e| < 2^100; zero below 2^-74.
__device__ __forceinline__ F2 f2_split_scaled(double x, int e) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int a = (int)(hi & 0x7FFFFFFFu) - (e << 20);
    const unsigned b = (__funnelshift_l(lo, (unsigned)a, 3) + 0x40000000u) | (hi & 0x80000000u);
    const bool tiny = a < ((1023 - 74) << 20);
    F2 r;
    r.h = tiny ? 0.0f : __uint_as_float(b);
    r.l = __fmul_rn((float)(int)(lo & 0x1FFFFFFFu), __uint_as_float(tiny ? 0u : (b & 0xFF800000u) - (52u << 23)));
    return r;
}

// A pair times 2^e as a double; zero below 2^-100.
__device__ __forceinline__ double f2_double_scaled(const F2& v, int e) {
    const F2 n = f2_norm(v.h, v.l);
    const double d = f2_double(n);
    return fabsf(n.h) < 7.8886091e-31f ? 0.0 : ldexp_bits(d, e);
}

__device__ __forceinline__ F2 f2_neg(const F2& a) { return F2{-a.h, -a.l}; }
__device__ __forceinline__ F2 f2_times(float k, const F2& a) { return f2_mul(F2{k, 0.0f}, a); }
// 1 + x for |x| < 1
__device__ __forceinline__ F2 f2_one_plus(const F2& x) {
    F2 r;
    fast_two_sum(1.0f, x.h, r.h, r.l);
    r.l = __fadd_rn(r.l, x.l);
    return r;
}

// What the tangent and the adjoint take from a drift's scalars.
struct DriftJac {
    F2 g0, g1, iD, p, j, y, X;
    F2 g4, g5, S;
    F2 hb0, hb1, hb2, hb3, Tb;  // -2 gb_n, -2 Tb
    F2 u;                       // dt mu / r0^5
    double tide;                // the same, FP64
};

__device__ __forceinline__ void drift_jac(const DriftSeries& s, DriftJac& o) {
    o.p = f2_one_plus(s.k);
    o.g1 = f2_one_plus(f2_neg(s.T));
    const F2 one = {1.0f, 0.0f};
    o.iD = f2_div(one, s.D, s.rD);
    const F2 bg2 = f2_mul(s.b, s.g2);
    o.g0 = f2_one_plus(f2_neg(bg2));
    o.j = f2_neg(f2_mul(f2_add(bg2, s.rho), o.iD));
    const F2 ap = f2_mul(s.a, o.p);
    const F2 t1 = f2_add(ap, f2_mul(o.j, ap));
    o.y = f2_sub(f2_sub(o.j, t1), f2_mul(s.q, f2_mul(o.p, o.p)));
    o.X = f2_add(f2_times(3.0f, s.k), f2_mul(o.p, f2_add(o.y, o.j)));
    const F2 S = f2_norm(s.S, s.d);
    o.S = S;
    const F2 S2 = f2_mul(S, S), S4 = f2_mul(S2, S2);
    const float z = s.b.h * S2.h;
    // c4 = 1/24 - z/720 + z^2/40320, c5 = 1/120 - z/5040 + z^2/362880 (terms in z: 2^-24 of 2^-13)
    F2 c4, c5;
    fast_two_sum(0.0416666679f, z * __fmaf_rn(z, 1.0f / 40320.0f, -1.0f / 720.0f), c4.h, c4.l);
    c4.l = __fadd_rn(c4.l, -1.24176334e-9f);
    fast_two_sum(0.00833333377f, z * __fmaf_rn(z, 1.0f / 362880.0f, -1.0f / 5040.0f), c5.h, c5.l);
    c5.l = __fadd_rn(c5.l, -4.34617164e-10f);
    const F2 g4 = f2_mul(S4, c4), g5 = f2_mul(f2_mul(S4, S), c5);
    o.g4 = g4;
    o.g5 = g5;
    o.hb0 = f2_mul(S, o.g1);
    o.hb1 = f2_sub(f2_mul(S, s.g2), s.g3);
    o.hb2 = f2_sub(f2_mul(S, s.g3), F2{2.0f * g4.h, 2.0f * g4.l});
    o.hb3 = f2_sub(f2_mul(S, g4), f2_times(3.0f, g5));
    o.Tb = f2_add(f2_add(o.hb1, f2_mul(s.a, o.hb2)), f2_mul(s.m, o.hb3));
    o.u = f2_mul(s.dts2, s.w);
    o.tide = s.dts * s.wd;
}

// The tide's factor times the FP64 dot product x: (dt mu / r0^5) x (3 + X).
__device__ __forceinline__ double tide_of(const DriftJac& J, double x) {
    return (J.tide * x) * (3.0 + f2_double(f2_norm(J.X.h, J.X.l)));
}

// t <- M t, M the drift's Jacobian at the state pre (pairs X, V); e = scale_exponent(t).
__device__ __forceinline__ void drift_tangent_split(const F2& dt2, const DriftSeries& s, const DriftFactors& f,
                                                    const DriftJac& J, const double (&pre)[6], const F2 (&X)[3],
                                                    const F2 (&V)[3], double (&t)[6], int e) {
    F2 R[3], W[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        R[c] = f2_split_scaled(t[c], e);
        W[c] = f2_split_scaled(t[3 + c], e);
    }
    const double x = fma(pre[0], t[0], fma(pre[1], t[1], pre[2] * t[2]));
    const double A = tide_of(J, x);
    const F2 al = f2_mul(s.w, f2_split_scaled(x, e));
    const F2 dw = f2_mul(dt2, s.w);
    const F2 eta = f2_mul(dw, f2_add(f2_dot(R, V), f2_dot(X, W)));
    const F2 zeta = f2_add(f2_mul(s.m, al), f2_mul(f2_mul(dt2, dw), f2_dot(V, W)));
    // dS = -p alpha + sn; dg_n in -2 gb_n zeta = hb_n zeta
    const F2 sn = f2_neg(f2_mul(f2_add(f2_mul(J.Tb, zeta), f2_mul(s.g2, eta)), J.iD));
    const F2 S = f2_sub(sn, f2_mul(J.p, al));
    const F2 dg2 = f2_add(f2_mul(J.g1, S), f2_mul(J.hb2, zeta));
    const F2 dg3 = f2_add(f2_mul(s.g2, S), f2_mul(J.hb3, zeta));
    // the parts of dg1 and theta without alpha's own
    const F2 bg1 = f2_mul(s.b, J.g1);
    const F2 n1 = f2_add(f2_mul(J.g0, sn), f2_mul(J.hb1, zeta));
    const F2 n2 = f2_add(f2_mul(J.g1, sn), f2_mul(J.hb2, zeta));
    const F2 n0 = f2_sub(f2_mul(J.hb0, zeta), f2_mul(bg1, sn));
    const F2 thn = f2_add(f2_add(n0, f2_mul(eta, J.g1)), f2_add(f2_mul(s.a, n1), f2_mul(s.m, n2)));
    // alpha's part of theta / D is (g0 / D)(1 - a p) - q p^2 = 1 + y
    const F2 thD = f2_add(f2_add(al, f2_mul(J.y, al)), f2_mul(thn, J.iD));
    const F2 cf = f2_sub(f2_mul(s.g2, al), dg2);                                        // df / m
    const F2 cd = f2_mul(J.iD, f2_sub(f2_mul(s.g2, thD), dg2));                          // dgdot / m
    const F2 cn = f2_mul(J.iD, f2_sub(f2_mul(J.p, thn), n1));  // dfdot dt / m without alpha's
    const F2 mf = f2_mul(s.m, cf), mg = f2_neg(f2_mul(f2_mul(dt2, s.m), dg3)), mn = f2_mul(s.dts2, cn),
             md = f2_mul(s.m, cd);
    double o[6];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const F2 a = f2_add(f2_add(f2_mul(s.fm1, R[c]), f2_mul(mf, X[c])), f2_mul(mg, V[c]));
        const F2 b = f2_add(f2_add(f2_mul(f.gdm1, W[c]), f2_mul(mn, X[c])), f2_mul(md, V[c]));
        o[c] = fma(f.g, t[3 + c], t[c]) + f2_double_scaled(a, e);
        o[3 + c] = fma(f.fd, t[c], fma(A, pre[c], t[3 + c])) + f2_double_scaled(b, e);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) t[c] = o[c];
}

// l <- M^T l: the reverse sweep through the same relations, with the cotangents of
// f, dg, dfdot, dgdot multiplied by dt (lf = dt lr.r, lg = dt^2 lr.v, P = lv.r, ld = dt lv.v).
__device__ __forceinline__ void drift_adjoint_split(const F2& dt2, const DriftSeries& s, const DriftFactors& f,
                                                    const DriftJac& J, const double (&pre)[6], const F2 (&X)[3],
                                                    const F2 (&V)[3], double (&l)[6], int e) {
    F2 R[3], W[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        R[c] = f2_split_scaled(l[c], e);
        W[c] = f2_split_scaled(l[3 + c], e);
    }
    const double x = fma(pre[0], l[3], fma(pre[1], l[4], pre[2] * l[5]));
    const double A = tide_of(J, x);
    const F2 P = f2_split_scaled(x, e);
    const F2 lf = f2_mul(dt2, f2_dot(R, X));
    const F2 lg = f2_mul(dt2, f2_mul(dt2, f2_dot(R, V)));
    const F2 tL = f2_mul(J.iD, f2_mul(dt2, f2_dot(W, V)));
    const F2 th = f2_mul(f2_mul(J.iD, s.g2), tL);  // theta's cotangent but for P's
    const F2 lfL = f2_add(lf, tL);
    // S's cotangent: sg without P's part, which is -(1 + y), sP with it; both over D: eg, eP
    const F2 sg = f2_sub(f2_mul(th, f2_add(f2_mul(s.a, J.g0), f2_mul(s.q, J.g1))),
                         f2_add(f2_mul(J.g1, lfL), f2_mul(s.g2, lg)));
    const F2 sP = f2_sub(f2_sub(sg, P), f2_mul(P, J.y));
    const F2 eg = f2_mul(J.iD, sg), eP = f2_mul(J.iD, sP);
    const F2 PiD = f2_mul(P, J.iD);
    const F2 ct = f2_add(th, f2_mul(PiD, J.p));
    const F2 c1 = f2_sub(f2_mul(s.a, ct), PiD);
    const F2 c2 = f2_sub(f2_mul(s.m, ct), lfL);
    const F2 H = f2_sub(f2_sub(f2_add(f2_add(f2_mul(J.hb0, ct), f2_mul(J.hb1, c1)), f2_mul(J.hb2, c2)),
                               f2_mul(J.hb3, lg)),
                        f2_mul(J.Tb, eP));
    // without P (3 + X): the tide's
    const F2 ca = f2_add(f2_add(f2_mul(s.g2, lf), f2_sub(f2_mul(J.g0, th), f2_mul(J.g1, eg))), f2_mul(s.m, H));
    const F2 ce = f2_sub(f2_mul(J.g1, ct), f2_mul(s.g2, eP));
    const F2 ua = f2_mul(J.u, ca), ue = f2_mul(f2_mul(dt2, J.u), ce), uk = f2_mul(f2_mul(dt2, f2_mul(dt2, J.u)), H);
    double o[6];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const F2 a = f2_add(f2_add(f2_mul(s.fm1, R[c]), f2_mul(ua, X[c])), f2_mul(ue, V[c]));
        const F2 b = f2_add(f2_add(f2_mul(f.gdm1, W[c]), f2_mul(ue, X[c])), f2_mul(uk, V[c]));
        o[c] = fma(f.fd, l[3 + c], fma(A, pre[c], l[c])) + f2_double_scaled(a, e);
        o[3 + c] = fma(f.g, l[c], l[3 + c]) + f2_double_scaled(b, e);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) l[c] = o[c];
}

// A pair and its derivative along a tangent, both pairs.
struct D2 {
    F2 v, d;
};
__device__ __forceinline__ D2 operator+(const D2& a, const D2& b) { return D2{f2_add(a.v, b.v), f2_add(a.d, b.d)}; }
__device__ __forceinline__ D2 operator-(const D2& a, const D2& b) { return D2{f2_sub(a.v, b.v), f2_sub(a.d, b.d)}; }
__device__ __forceinline__ D2 operator*(const D2& a, const D2& b) {
    return D2{f2_mul(a.v, b.v), f2_add(f2_mul(a.v, b.d), f2_mul(a.d, b.v))};
}
__device__ __forceinline__ D2 operator*(float k, const D2& a) { return D2{f2_times(k, a.v), f2_times(k, a.d)}; }

// The second derivative of the drift contracted with a tangent t = (Xi, Nu) and a cotangent
// (Lr, Lv), all scaled pairs: o = d(M^T l)[t].  drift_adjoint_split's relations,
// unreduced, with their derivatives: its terms are of first order in n dt and smaller, and
// added to a sum that already holds the same products of earlier steps, so
// that pairs serve all of them (to 2^-43 of the term against 113-bit differences).
__device__ __forceinline__ void drift_second_split(const F2& dt2, const DriftSeries& s, const DriftJac& J,
                                                   const F2 (&X)[3], const F2 (&V)[3], const F2 (&Xi)[3],
                                                   const F2 (&Nu)[3], const F2 (&Lr)[3], const F2 (&Lv)[3],
                                                   F2 (&o)[6]) {
    const F2 dw = f2_mul(dt2, s.w);
    const F2 al = f2_mul(s.w, f2_dot(X, Xi));
    const F2 eta = f2_mul(dw, f2_add(f2_dot(Xi, V), f2_dot(X, Nu)));
    const F2 kap = f2_mul(f2_mul(dt2, dw), f2_dot(V, Nu));
    const F2 zeta = f2_add(f2_mul(s.m, al), kap);
    const F2 sig = f2_neg(f2_mul(f2_add(f2_add(f2_mul(J.g1, al), f2_mul(s.g2, eta)), f2_mul(J.Tb, zeta)), J.iD));
    // -2 gb4, -2 gb5 (g6 = S^6 c6, g7 = S^7 c7)
    const float S6 = J.S.h * J.S.h * J.S.h * J.S.h * J.S.h * J.S.h;
    const float g6 = S6 * __fmaf_rn(s.b.h, -1.0f / 40320.0f, 1.0f / 720.0f), g7 = S6 * J.S.h * (1.0f / 5040.0f);
    const F2 hb4 = f2_sub(f2_mul(J.S, J.g5), F2{4.0f * g6, 0.0f});
    const F2 hb5 = {__fmaf_rn(J.S.h, g6, -5.0f * g7), 0.0f};
    const F2 e0 = f2_sub(f2_mul(J.hb0, zeta), f2_mul(f2_mul(s.b, J.g1), sig));
    const F2 e1 = f2_add(f2_mul(J.g0, sig), f2_mul(J.hb1, zeta));
    const F2 e2 = f2_add(f2_mul(J.g1, sig), f2_mul(J.hb2, zeta));
    const F2 e3 = f2_add(f2_mul(s.g2, sig), f2_mul(J.hb3, zeta));
    const F2 e4 = f2_add(f2_mul(s.g3, sig), f2_mul(hb4, zeta));
    const F2 e5 = f2_add(f2_mul(J.g4, sig), f2_mul(hb5, zeta));
    const F2 thD = f2_mul(J.iD, f2_add(f2_add(f2_mul(al, J.g0), e0),
                                       f2_add(f2_mul(eta, J.g1), f2_add(f2_mul(s.a, e1), f2_mul(s.m, e2)))));
    // the factors' derivatives
    const F2 adt = f2_add(thD, al);
    const F2 df = f2_mul(s.m, f2_sub(f2_mul(s.g2, al), e2));
    const F2 dg = f2_neg(f2_mul(f2_mul(dt2, s.m), e3));
    const F2 dfd = f2_mul(s.dts2, f2_sub(f2_mul(J.p, adt), f2_mul(J.iD, e1)));
    const F2 dgd = f2_mul(f2_mul(s.m, J.iD), f2_sub(f2_mul(s.g2, thD), e2));
    // total derivatives of the normalised scalars (h = dt / r0 changes too)
    const D2 S = {J.S, f2_add(sig, f2_mul(al, J.S))};
    const D2 g0 = {J.g0, e0}, g1 = {J.g1, f2_add(e1, f2_mul(al, J.g1))};
    const D2 g2 = {s.g2, f2_add(e2, f2_times(2.0f, f2_mul(al, s.g2)))};
    const D2 g3 = {s.g3, f2_add(e3, f2_times(3.0f, f2_mul(al, s.g3)))};
    const D2 g4 = {J.g4, f2_add(e4, f2_times(4.0f, f2_mul(al, J.g4)))};
    const D2 g5 = {J.g5, f2_add(e5, f2_times(5.0f, f2_mul(al, J.g5)))};
    const D2 a = {s.a, f2_sub(eta, f2_times(2.0f, f2_mul(al, s.a)))};
    const D2 m = {s.m, f2_times(-3.0f, f2_mul(al, s.m))};
    const D2 b = {s.b, f2_times(2.0f, f2_sub(f2_mul(al, f2_sub(s.q, f2_times(2.0f, s.m))), kap))};
    const D2 iD = {J.iD, f2_mul(J.iD, f2_sub(al, thD))};
    // the adjoint
    const F2 dtt = f2_mul(dt2, dt2);
    const D2 lf = {f2_mul(dt2, f2_dot(Lr, X)), f2_mul(dt2, f2_dot(Lr, Xi))};
    const D2 lg = {f2_mul(dtt, f2_dot(Lr, V)), f2_mul(dtt, f2_dot(Lr, Nu))};
    const D2 PiD = iD * D2{f2_dot(Lv, X), f2_dot(Lv, Xi)};
    const D2 tL = iD * D2{f2_mul(dt2, f2_dot(Lv, V)), f2_mul(dt2, f2_dot(Lv, Nu))};
    const D2 c0 = iD * (PiD * g1 + tL * g2);
    const D2 c1 = c0 * a - PiD;
    const D2 c2 = c0 * m - (lf + tL);
    const D2 e = iD * (g0 * c1 + g1 * (c2 - b * c0) - g2 * lg);
    const D2 hb1 = S * g2 - g3, hb2 = S * g3 - 2.0f * g4, hb3 = S * g4 - 3.0f * g5;
    const D2 H = S * g1 * c0 + hb1 * c1 + hb2 * c2 - hb3 * lg - (hb1 + a * hb2 + m * hb3) * e;
    const D2 ca = g2 * lf + g1 * (PiD - e) + g0 * c0 + m * H;
    const D2 ce = g1 * c0 - g2 * e;
    const D2 u = {J.u, f2_times(-5.0f, f2_mul(al, J.u))};
    const D2 ua = u * ca;
    const D2 ud = {f2_mul(dt2, u.v), f2_mul(dt2, u.d)}, ue = ud * ce;
    const D2 uk = D2{f2_mul(dt2, ud.v), f2_mul(dt2, ud.d)} * H;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        o[c] = f2_add(f2_add(f2_add(f2_mul(df, Lr[c]), f2_mul(dfd, Lv[c])),
                             f2_add(f2_mul(ua.d, X[c]), f2_mul(ua.v, Xi[c]))),
                      f2_add(f2_mul(ue.d, V[c]), f2_mul(ue.v, Nu[c])));
        o[3 + c] = f2_add(f2_add(f2_add(f2_mul(dg, Lr[c]), f2_mul(dgd, Lv[c])),
                                 f2_add(f2_mul(ue.d, X[c]), f2_mul(ue.v, Xi[c]))),
                          f2_add(f2_mul(uk.d, V[c]), f2_mul(uk.v, Nu[c])));
    }
}

// One planet's share of the tidal matrix of a full kick, dt A w = -s (w - 3 d (d.w) / |d|^2) with
// s = dt G m / |d|^3, added to acc (w: the scaled pairs W).  False, adding nothing, when
// the planet is near (as in kick_split): the caller then forms the term in FP64.
__device__ __forceinline__ bool kick_jac_split(const F2 (&x)[3], const F2 (&P)[3], const F2& tg, float lim2,
                                               const F2 (&W)[3], F2 (&acc)[3]) {
    F2 d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = f2_sub(x[c], P[c]);
    const RsqrtF2 r = f2_rsqrt(f2_norm2(d));
    F2 s = f2_k_rcube(r, tg);
    const bool far = s.h * s.h <= lim2;
    s.h = far ? s.h : 0.0f;
    s.l = far ? s.l : 0.0f;
    const F2 inv = {far ? r.yy : 0.0f, far ? __fmaf_rn(r.yy, r.e * __fadd_rn(1.0f, r.e), r.yl) : 0.0f};
    const F2 t = f2_mul(f2_mul(s, inv), f2_times(3.0f, f2_dot(d, W)));
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[c] = f2_add(acc[c], f2_sub(f2_mul(t, d[c]), f2_mul(s, W[c])));
    return far;
}

// The same for two cotangents W, U and the matrix's derivative along Xi applied to W,
//   d(dt A)[xi] w = 3 s (mu w + la xi + (xi.w / |d|^2 - 5 mu la) d),  mu = d.xi / |d|^2, la = d.w / |d|^2:
// accW, accU += dt A w, dt A u; accD += d(dt A)[xi] w.
__device__ __forceinline__ bool kick_second_split(const F2 (&x)[3], const F2 (&P)[3], const F2& tg, float lim2,
                                                  const F2 (&W)[3], const F2 (&U)[3], const F2 (&Xi)[3],
                                                  F2 (&accW)[3], F2 (&accU)[3], F2 (&accD)[3]) {
    F2 d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = f2_sub(x[c], P[c]);
    const RsqrtF2 r = f2_rsqrt(f2_norm2(d));
    F2 s = f2_k_rcube(r, tg);
    const bool far = s.h * s.h <= lim2;
    s.h = far ? s.h : 0.0f;
    s.l = far ? s.l : 0.0f;
    const F2 inv = {far ? r.yy : 0.0f, far ? __fmaf_rn(r.yy, r.e * __fadd_rn(1.0f, r.e), r.yl) : 0.0f};
    const F2 s3 = f2_times(3.0f, s);
    const F2 la = f2_mul(inv, f2_dot(d, W)), mu = f2_mul(inv, f2_dot(d, Xi));
    const F2 tw = f2_mul(s3, la), tu = f2_mul(s3, f2_mul(inv, f2_dot(d, U)));
    const F2 tm = f2_mul(s3, mu);
    const F2 td = f2_mul(s3, f2_sub(f2_mul(inv, f2_dot(Xi, W)), f2_times(5.0f, f2_mul(mu, la))));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        accW[c] = f2_add(accW[c], f2_sub(f2_mul(tw, d[c]), f2_mul(s, W[c])));
        accU[c] = f2_add(accU[c], f2_sub(f2_mul(tu, d[c]), f2_mul(s, U[c])));
        accD[c] = f2_add(accD[c], f2_add(f2_add(f2_mul(tm, W[c]), f2_mul(tw, Xi[c])), f2_mul(td, d[c])));
    }
    return far;
}

}  // namespace glisse
