// ephemeris.cu -- the planets: set-up and the chunked Wisdom-Holman map (section 2.2).
//
// The paper integrates the planets with the standard mixed-variable
// symplectic (Wisdom-Holman) map in Jacobi coordinates, a chunk of steps
// ahead of the particles, and ships the heliocentric positions plus the
// common indirect term h0 = -sum_j G m_j r_j / |r_j|^3 for every step.
// Here that runs on the GPU in one block of three warps on a side stream, one
// chunk ahead of the particle kernel: warp 0 steps the planets (its lanes are
// planet rows x 4 columns, so each pair interaction is computed once, in
// parallel lanes), warps 1 and 2 -- on other SM partitions -- turn every step's
// synchronised state into the log records with h0 and the heliocentric history.
//
// Jacobi coordinates (commented equations after Eq. 2 of the paper), planets
// i = 1..N_p (lane i-1), star 0:
//   eta_i = m0 + m_1 + ... + m_i
//   r'_i = r_i - sum_{k<i} m_k r_k / eta_{i-1}        (helio -> Jacobi)
//   r_i  = r'_i + sum_{k<i} (m_k / eta_k) r'_k         (Jacobi -> helio)
// Kepler part of H: sum_i p'_i^2 / 2m'_i - G m0 m_i / |r'_i| with
//   m'_i = m_i eta_{i-1} / eta_i, i.e. a Kepler drift with mu_i = G m0 eta_i / eta_{i-1}.
// Interaction part: H_int = sum_i G m0 m_i (1/|r'_i| - 1/|r_i|) - sum_{i<j} G m_i m_j / |r_i - r_j|.
// Its kick, by the chain rule through r(r'):
//   dv'_k/dt = -(eta_k / eta_{k-1}) [ -G m0 r'_k / |r'_k|^3 + ghat_k + S_k / eta_k ]
//   ghat_i = G m0 r_i / |r_i|^3 + sum_{j != i} G m_j (r_i - r_j) / |r_i - r_j|^3
//   S_k = sum_{i > k} m_i ghat_i
#include "glisse_internal.h"
#include "kepler.cuh"
#include "split_math.cuh"

namespace glisse {

// One log record: (x, y, z) as doubles, (sx, sy, sz) as pairs (the same vector, or dt times it).
__device__ __forceinline__ void store_rec(double* __restrict__ rec, double x, double y, double z, double sx, double sy,
                                          double sz) {
    const F2 a = f2_split(sx), b = f2_split(sy), c = f2_split(sz);
    reinterpret_cast<double2*>(rec)[0] = make_double2(x, y);
    reinterpret_cast<double2*>(rec)[1] = make_double2(z, 0.0);
    reinterpret_cast<float4*>(rec + kRecSplit)[0] = make_float4(a.h, b.h, c.h, a.l);
    reinterpret_cast<float4*>(rec + kRecSplit)[1] = make_float4(b.l, c.l, 0.0f, 0.0f);
}

// Scans over the first n lanes (n <= 32, warp-uniform).  Lanes >= n must hold 0.
// exclusive prefix: sum over lanes k < lane
__device__ __forceinline__ double warp_excl_prefix(double v, int lane, int n) {
    double incl = v;
    for (int o = 1; o < n; o <<= 1) {
        const double t = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += t;
    }
    return incl - v;
}

// ---------------------------------------------------------------------------
// Set-up: constants, Jacobi state, encounter radii.  One warp.
//   planets : [np][7] heliocentric m, x, y, z, vx, vy, vz (device copy)
//   jac     : out [2][np][3]: Jacobi positions then Jacobi velocities
//   status  : out 0, or GLISSE_E_INVAL (unbound planet, or not ordered by a)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(32) eph_setup_kernel(const double* __restrict__ planets, int np, double m0, double G,
                                                         int enc_mode, double enc_value, PlanetConsts* pc,
                                                         double* jac, int* status) {
    const int lane = threadIdx.x;
    const bool on = lane < np;
    const double m = on ? planets[7 * lane] : 0.0;
    double r[3], v[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        r[d] = on ? planets[7 * lane + 1 + d] : 0.0;
        v[d] = on ? planets[7 * lane + 4 + d] : 0.0;
    }
    // eta_i for this lane's planet (inclusive) and eta_{i-1}
    const double eta_prev = m0 + warp_excl_prefix(m, lane, 32);
    const double eta_i = eta_prev + m;
    double q[3], w[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double mr = warp_excl_prefix(m * r[d], lane, 32);
        const double mv = warp_excl_prefix(m * v[d], lane, 32);
        q[d] = r[d] - mr / eta_prev;
        w[d] = v[d] - mv / eta_prev;
    }
    // initial osculating heliocentric semi-major axis with mu = G (m0 + m_j)
    const double rn = sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
    const double v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    const double inva = 2.0 / rn - v2 / (G * (m0 + m));
    const bool bound = inva > 0.0;
    const double a = 1.0 / inva;
    const double rcrit = (enc_mode == GLISSE_ENC_FIXED) ? enc_value : enc_value * a * cbrt(m / (3.0 * m0));
    // ordering by increasing a
    const double a_prev = __shfl_up_sync(kFullMask, a, 1);
    const bool order_ok = (lane == 0) || !(a <= a_prev);
    const unsigned bad = __ballot_sync(kFullMask, on && (!bound || !order_ok || !isfinite(rcrit)));
    if (on) {
        pc->m[lane] = m;
        pc->eta[lane + 1] = eta_i;
        pc->mu_jac[lane] = G * m0 * eta_i / eta_prev;
        pc->gm[lane] = G * m;
        pc->rcrit[lane] = rcrit;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            jac[3 * lane + d] = q[d];
            jac[3 * np + 3 * lane + d] = w[d];
        }
    }
    if (lane == 0) {
        pc->np = np;
        pc->m0 = m0;
        pc->G = G;
        pc->mu0 = G * m0;
        pc->eta[0] = m0;
        *status = bad ? GLISSE_E_INVAL : 0;
    }
}

// ---------------------------------------------------------------------------
// The chunked Wisdom-Holman step of the planets.
//
// The steps are serial and one warp takes them, so a step lasts as long as its
// chain of dependent instructions: 64 cycles for each FP64 one whatever the
// lanes doing it, ~4 for an FP32 one, ~30 for a shuffle.  What shortens it:
//   * warp 0 holds planet i in the four lanes 4i .. 4i + 3.  The drift's FP64
//     arithmetic is the fast path of kepler.cuh with each instruction doing
//     different things in a row's lanes (u and v^2; c2 and c3; F and r; the three
//     components of x and v; ...): 31 FP64 instructions instead of ~66;
//   * the kick is ~1e-3 of the velocity and is formed in float pairs
//     (split_math.cuh) with lane 4i + c taking the interaction with planet j = c
//     (and c + 4 for 5 to 8 planets); the star's part, which nearly cancels between
//     Jacobi and heliocentric positions, is taken as the small difference itself;
//   * what only the log needs runs on other SM partitions from a double-buffered
//     shared-memory hand-off ordered by named barriers: warp 1 writes the log
//     records (positions, h0) and the progress count, warp 2 the synchronised
//     heliocentric states.
// Each step is open half kick, Kepler drift of every Jacobi body, positions,
// kick terms, closing half kick, identically at every step, so the planet
// sequence does not depend on where chunks begin.
// ---------------------------------------------------------------------------
constexpr int kEphCols = 4;     // lanes per planet row in warp 0
constexpr int kStopEvery = 16;  // steps between looks at the stop word

// named barriers of the hand-off ring: FULL slot b = 1 + b, EMPTY slot b = 3 + b,
// 5: warps 1 and 2 before a progress count
__device__ __forceinline__ void eph_bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void eph_bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

struct EphRing {
    double q[2][kMaxPlanets][3];  // Jacobi positions of the emitted step
    double w[2][kMaxPlanets][3];  // synchronised Jacobi velocities
    F2 d[2][kMaxPlanets][3];      // heliocentric minus Jacobi position
    int stop;                     // warp 1 saw the stop word
    int last[2];                  // warp 0: nothing comes in this slot, or after it
};

// Sum over the four lanes of a planet row (every lane of the row gets the same bits).
__device__ __forceinline__ double row_sum(double v) {
    v += __shfl_xor_sync(kFullMask, v, 1);
    v += __shfl_xor_sync(kFullMask, v, 2);
    return v;
}

__device__ __forceinline__ F2 shfl_f2(const F2& v, int src) {
    return F2{__shfl_sync(kFullMask, v.h, src), __shfl_sync(kFullMask, v.l, src)};
}

__device__ __forceinline__ F2 row_sum(F2 v) {
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1)
        v = f2_add(v, F2{__shfl_xor_sync(kFullMask, v.h, o), __shfl_xor_sync(kFullMask, v.l, o)});
    return v;
}

// Column c's value in the lane's row.
__device__ __forceinline__ double row_bc(double v, int c) { return __shfl_sync(kFullMask, v, c, kEphCols); }

// Warp 0: positions r from the Jacobi positions q of every row (r_i = q_i + sum_{k<i} m_k/eta_k q_k).
template <int H>
__device__ __forceinline__ void eph_positions(const double (&moe)[2], const bool (&below)[2], const double q[3],
                                              double r[3], int col) {
    double p[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int src = kEphCols * (col + kEphCols * h);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double qj = __shfl_sync(kFullMask, q[d], src);
            p[d] = fma(below[h] ? moe[h] : 0.0, qj, p[d]);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) r[d] = q[d] + row_sum(p[d]);
}

// Warp 0: Jacobi acceleration of the row's planet at heliocentric positions r.
//   ghat_i = G m0 r_i / |r_i|^3 + sum_{j != i} G m_j (r_i - r_j) / |r_i - r_j|^3  (lane-parallel over j)
//   S_k    = sum_{i > k} m_i ghat_i                                             (lane-parallel over i)
//   acc_k  = -(eta_k / eta_{k-1}) [ghat_k + S_k / eta_k - G m0 q_k / |q_k|^3]
template <int H>
__device__ __forceinline__ void eph_accel(const PlanetConsts& pc, bool on, int row, int col, const double (&kj)[2],
                                          const bool (&valid)[2], const double (&mi)[2], const bool (&above)[2],
                                          double inv_eta, double ratio, const double q[3], double qr,
                                          const double r[3], double acc[3]) {
    double t[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int j = col + kEphCols * h;
        const int src = kEphCols * j;
        const bool self = j == row;
        double dv[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double rj = __shfl_sync(kFullMask, r[d], src);
            dv[d] = r[d] - (self ? 0.0 : rj);
        }
        const double d2 = fma(dv[0], dv[0], fma(dv[1], dv[1], dv[2] * dv[2]));
        const double sc = k_rcube(valid[h] ? d2 : 1.0, kj[h]);
#pragma unroll
        for (int d = 0; d < 3; ++d) t[d] = fma(sc, dv[d], t[d]);
    }
    double gh[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) gh[d] = row_sum(t[d]);
    double sv[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int src = kEphCols * (col + kEphCols * h);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double gi = __shfl_sync(kFullMask, gh[d], src);
            sv[d] = fma(above[h] ? mi[h] : 0.0, gi, sv[d]);
        }
    }
    // |q|^2 from the radius the drift leaves (or radius_of at a chunk's start: the same expression)
    const double iq3 = k_rcube(on ? qr * qr : 1.0, pc.mu0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double S = row_sum(sv[d]);
        const double grad = fma(S, inv_eta, fma(-iq3, q[d], gh[d]));
        acc[d] = on ? -ratio * grad : 0.0;
    }
}

// What a lane of warp 0 keeps for the kick.  Per column j = col + 4h: m_j / eta_j for the
// positions (j < row), the kick's G-coefficient (G m0 on the diagonal, G m_j off it),
// m_j for the suffix sums (j > row); zero where the lane has no such term.
struct EphLane {
    int row, col;
    bool on;
    bool valid[2];
    F2 moe[2], kj[2], mi[2], inv_eta, ratio_dt, gm0;
    bool light;  // every planet below 2^-7 of the star's mass
};

// Limits of the pairs' kick: s = dt G m_j / |d|^3 against the orbit's rate (as in kick_split),
// and |r|^2 / |q|^2 - 1 of the heliocentric and Jacobi positions.
constexpr float kEphNear2 = 1.6e-5f;  // (0.004)^2
constexpr float kEphEps = 0.015625f;

// The kick of a full step, dt dv/dt, for component min(col, 2) of the row's planet, at Jacobi
// positions q; delta: heliocentric minus Jacobi position.
//   a_i = ghat_i - G m0 q_i / |q_i|^3
//       = sum_{j != i} G m_j (r_i - r_j) / |r_i - r_j|^3 + G m0 |r_i|^-3 (delta_i - Y q_i),
//   Y = (|r|/|q|)^3 - 1 = e (3 + 3e + e^2) / (1 + X), e = |r|^2/|q|^2 - 1, X = |r|^3/|q|^3,
//   dv'_k/dt = -(eta_k / eta_{k-1}) [a_k + S_k / eta_k], S_k = sum_{i>k} m_i (a_i + G m0 q_i/|q_i|^3).
// Returns false (on every lane) where a term is too large for pairs.
template <int H>
__device__ __forceinline__ bool eph_kick(const EphLane& ln, const double q[3], F2 (&delta)[3], double& K) {
    const F2 Q[3] = {f2_split(q[0]), f2_split(q[1]), f2_split(q[2])};
    F2 t[3] = {F2{0.f, 0.f}, F2{0.f, 0.f}, F2{0.f, 0.f}};
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int src = kEphCols * (ln.col + kEphCols * h);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const F2 p = f2_mul(ln.moe[h], shfl_f2(Q[d], src));
            t[d] = h == 0 ? p : f2_add(t[d], p);
        }
    }
    F2 R[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        delta[d] = row_sum(t[d]);
        R[d] = f2_add(Q[d], delta[d]);
    }
    // |q|^-3 G m0, and Y's e = (2 q + delta) . delta / |q|^2
    const RsqrtF2 iq = f2_rsqrt(f2_norm2(Q));
    const F2 cq = f2_k_rcube(iq, ln.gm0);
    const float rate2 = cq.h;  // G m0 / |q|^3: the orbit's rate squared
    F2 q2d[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) q2d[d] = f2_add(F2{2.0f * Q[d].h, 2.0f * Q[d].l}, delta[d]);
    const F2 w = F2{iq.yy, __fmaf_rn(iq.yy, __fmaf_rn(iq.e, iq.e, iq.e), iq.yl)};
    const F2 e = f2_mul(f2_dot(q2d, delta), w);
    bool fine = ln.light && fabsf(e.h) <= kEphEps;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int j = ln.col + kEphCols * h;
        const int src = kEphCols * j;
        const bool self = j == ln.row;
        F2 dv[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const F2 Rj = shfl_f2(R[d], src);
            dv[d] = self ? R[d] : f2_sub(R[d], Rj);
        }
        F2 D = f2_norm2(dv);
        if (!ln.valid[h]) D = F2{1.f, 0.f};
        const F2 s = f2_k_rcube(f2_rsqrt(D), ln.kj[h]);
        if (self) {
            const F2 X = f2_div(cq, s, rcp_f32(s.h));
            const F2 X1 = f2_add(F2{1.f, 0.f}, X);
            const F2 p = f2_mul(e, f2_add(F2{3.f, 0.f}, f2_mul(e, f2_add(F2{3.f, 0.f}, e))));
            const F2 Y = f2_div(p, X1, rcp_f32(X1.h));
#pragma unroll
            for (int d = 0; d < 3; ++d) dv[d] = f2_fnma(Y, Q[d], delta[d]);
        } else {
            fine = fine && (!ln.valid[h] || s.h * s.h * (ln.ratio_dt.h * ln.ratio_dt.h) <= kEphNear2 * rate2);
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const F2 p = f2_mul(s, dv[d]);
            t[d] = h == 0 ? p : f2_add(t[d], p);
        }
    }
    F2 a[3], g[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        a[d] = row_sum(t[d]);
        g[d] = ln.on ? f2_add(a[d], f2_mul(cq, Q[d])) : F2{0.f, 0.f};
    }
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int src = kEphCols * (ln.col + kEphCols * h);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const F2 p = f2_mul(ln.mi[h], shfl_f2(g[d], src));
            t[d] = h == 0 ? p : f2_add(t[d], p);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) t[d] = row_sum(t[d]);
    // this lane's component
    const F2 ac = ln.col == 0 ? a[0] : (ln.col == 1 ? a[1] : a[2]);
    const F2 Sc = ln.col == 0 ? t[0] : (ln.col == 1 ? t[1] : t[2]);
    const F2 k = f2_mul(ln.ratio_dt, f2_add(ac, f2_mul(ln.inv_eta, Sc)));
    K = ln.on ? f2_double(f2_norm(-k.h, -k.l)) : 0.0;
    return __all_sync(kFullMask, fine || !ln.on);
}

// eph_kick in FP64 (eph_positions, eph_accel), for the steps it leaves.  qr = |q|.
template <int H>
__device__ __noinline__ void eph_kick_fp64(const PlanetConsts& pc, double dt, double q0, double q1, double q2,
                                           double qr, F2 (&delta)[3], double& K) {
    const int np = pc.np;
    const int row = (threadIdx.x & 31) / kEphCols, col = threadIdx.x % kEphCols;
    const bool on = row < np;
    double moe[2], kj[2], mi[2];
    bool below[2], valid[2], above[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = col + kEphCols * h;
        const bool jon = h < H && j < np;
        below[h] = jon && on && j < row;
        above[h] = jon && on && j > row;
        valid[h] = jon && on;
        moe[h] = jon ? pc.m[j] / pc.eta[j + 1] : 0.0;
        kj[h] = valid[h] ? (j == row ? pc.mu0 : pc.gm[j]) : 0.0;
        mi[h] = jon ? pc.m[j] : 0.0;
    }
    const double inv_eta = on ? 1.0 / pc.eta[row + 1] : 1.0;
    const double ratio = on ? pc.eta[row + 1] / pc.eta[row] : 1.0;
    const double q[3] = {q0, q1, q2};
    double r[3], acc[3];
    eph_positions<H>(moe, below, q, r, col);
    eph_accel<H>(pc, on, row, col, kj, valid, mi, above, inv_eta, ratio, q, qr, r, acc);
    K = dt * (col == 0 ? acc[0] : (col == 1 ? acc[1] : acc[2]));
#pragma unroll
    for (int d = 0; d < 3; ++d) delta[d] = f2_split(r[d] - q[d]);
}

// eph_kick, or eph_kick_fp64 for the steps it leaves (its results through temporaries, so
// that the usual ones stay in registers).
template <int H>
__device__ __forceinline__ void eph_kick_any(const PlanetConsts& pc, const EphLane& ln, double dt, const double q[3],
                                             double qr, F2 (&delta)[3], double& K) {
    if (!eph_kick<H>(ln, q, delta, K)) {
        F2 d[3];
        double k;
        eph_kick_fp64<H>(pc, dt, q[0], q[1], q[2], qr, d, k);
        delta[0] = d[0];
        delta[1] = d[1];
        delta[2] = d[2];
        K = k;
    }
}

// Warp 0: hand an emitted step to the other warps in slot b.
__device__ __forceinline__ void eph_hand_over(EphRing& ring, const EphLane& ln, int b, double qc, double wc,
                                              const F2 (&delta)[3], int threads) {
    if (ln.on && ln.col < 3) {
        ring.q[b][ln.row][ln.col] = qc;
        ring.w[b][ln.row][ln.col] = wc;
        ring.d[b][ln.row][ln.col] = ln.col == 0 ? delta[0] : (ln.col == 1 ? delta[1] : delta[2]);
    }
    eph_bar_arrive(1 + b, threads);
}

// Warp 0 of the block: nsteps steps from the Jacobi state `jac` (in place), each step's
// synchronised state handed to the other warps.  status: GLISSE_E_KEPLER if a planet's
// drift fails.  threads: of the block.
template <int H>
__device__ __forceinline__ void eph_dynamics(const PlanetConsts& pc, double* jac, double dt, int nsteps, EphRing& ring,
                                             int* status, int threads) {
    const int np = pc.np;
    const int lane = threadIdx.x & 31;
    EphLane ln;
    ln.row = lane / kEphCols;
    ln.col = lane % kEphCols;
    ln.on = ln.row < np;
    const int row = ln.row, col = ln.col;
    const bool on = ln.on, odd = (col & 1) != 0;
    double q[3], w[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        q[d] = on ? jac[3 * row + d] : (d == 0 ? 1.0 + row : 0.0);
        w[d] = on ? jac[3 * np + 3 * row + d] : 0.0;
    }
    ln.inv_eta = f2_const(on ? 1.0 / pc.eta[row + 1] : 1.0);
    ln.ratio_dt = f2_const(on ? dt * (pc.eta[row + 1] / pc.eta[row]) : 0.0);
    ln.gm0 = f2_const(pc.mu0);
    const double mu = on ? pc.mu_jac[row] : pc.mu0;
    const float muf = d2f_bits(mu), dtf = d2f_bits(dt);
    ln.light = true;
    for (int j = 0; j < np; ++j) ln.light = ln.light && pc.m[j] <= 0.0078125 * pc.m0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = col + kEphCols * h;
        const bool jon = h < H && j < np;
        ln.valid[h] = jon && on;
        ln.moe[h] = f2_const(jon && on && j < row ? pc.m[j] / pc.eta[j + 1] : 0.0);
        ln.kj[h] = f2_const(ln.valid[h] ? (j == row ? pc.mu0 : pc.gm[j]) : 0.0);
        ln.mi[h] = f2_const(jon && on && j > row ? pc.m[j] : 0.0);
    }

    // |q| and mu/|q| of the Jacobi position: here from the position, then from each drift
    // (the same expressions)
    double r0, mur0, K;
    radius_of(q[0], q[1], q[2], r0, mur0);
    mur0 *= mu;
    F2 delta[3];
    eph_kick_any<H>(pc, ln, dt, q, r0, delta, K);
    const auto own = [col](const double (&a)[3]) { return col == 0 ? a[0] : (col == 1 ? a[1] : a[2]); };
    double wc = own(w);
    eph_hand_over(ring, ln, 0, own(q), wc, delta, threads);
    bool failed = false;
    for (int k = 0; k < nsteps; ++k) {
        // opening half kick
        wc = fma(0.5, K, wc);
#pragma unroll
        for (int d = 0; d < 3; ++d) w[d] = row_bc(wc, d);
        // ---- Kepler drift: the fast path of kepler.cuh, its FP64 work spread over the row's lanes ----
        const double dot = fma(col == 0 ? q[0] : w[0], w[0],
                               fma(col == 0 ? q[1] : w[1], w[1], (col == 0 ? q[2] : w[2]) * w[2]));
        const double u = row_bc(dot, 0), v2 = row_bc(dot, 1);
        // beta = 2 mu/r0 - v^2, qq = mu - beta r0 = v^2 r0 - mu
        const double bq = fma(odd ? v2 : 2.0, odd ? r0 : mur0, odd ? -mu : -v2);
        const double beta = row_bc(bq, 0), qq = row_bc(bq, 1);
        const float r0f = d2f_bits(r0), uf = d2f_bits(u), bf = d2f_bits(beta), qf = d2f_bits(qq);
        const int er = exp_bits(r0), ev = exp_bits(v2);
        bool ok = er > 1023 - 60 && er < 1023 + 60 && ev < 1023 + 120 && ev > 1023 - 200;
        float sf, dsf = 0.f;
        {
            // start: the series of s in dt to the third order; then Newton steps, two for nearly
            // circular orbits, until every planet's is below 2^-20 (five at most)
            const float ir = rcp_f32(r0f), h = dtf * ir, a = uf * h * ir;
            sf = h * fmaf(-1.0f / 6.0f * qf * ir, h * h, fmaf(0.5f * a, a - 1.0f, 1.0f));
        }
#pragma unroll 1
        for (int it = 0; it < 5; ++it) {
            const float s2f = sf * sf, zf = bf * s2f;
            const float c2 =
                fmaf(zf, fmaf(zf, fmaf(zf, -1.0f / 40320.0f, 1.0f / 720.0f), -1.0f / 24.0f), 0.5f);
            const float c3 =
                fmaf(zf, fmaf(zf, fmaf(zf, -1.0f / 362880.0f, 1.0f / 5040.0f), -1.0f / 120.0f), 1.0f / 6.0f);
            const float G1 = sf * fmaf(-zf, c3, 1.0f), G2 = s2f * c2, G3 = s2f * sf * c3;
            const float F = fmaf(r0f, G1, fmaf(uf, G2, fmaf(muf, G3, -dtf)));
            const float Fp = fmaf(r0f, fmaf(-zf, c2, 1.0f), fmaf(uf, G1, muf * G2));
            dsf = -F * rcp_f32(Fp);
            sf += dsf;
            if (it >= 1 && __all_sync(kFullMask, !on || fabsf(dsf) <= 9.5367431640625e-7f * fabsf(sf))) break;
        }
        const float zf = bf * sf * sf;
        ok = ok && fabsf(zf) <= kZ7 && fabsf(dsf) <= 9.5367431640625e-7f * fabsf(sf) && isfinite(sf);
        const double s0 = f2d_bits(sf);
        double s2, s3;
        ok = float_powers(sf, s2, s3) && ok;
        const double z = beta * s2;
        // c2 (even columns) and c3: four FP64 levels over a float tail (z^4 / 10! and beyond)
        double p;
        {
            const float t2 = fmaf(zf, fmaf(zf, -1.0f / 20922789888000.0f, 1.0f / 87178291200.0f), -1.0f / 479001600.0f);
            const float t3 = fmaf(zf, fmaf(zf, -1.0f / 355687428096000.0f, 1.0f / 1307674368000.0f),
                                  -1.0f / 6227020800.0f);
            const float tail = fmaf(zf, odd ? t3 : t2, odd ? 1.0f / 39916800.0f : 1.0f / 3628800.0f);
            p = fma(f2d_bits(tail), z, odd ? -1.0 / 362880.0 : -1.0 / 40320.0);
            p = fma(p, z, odd ? 1.0 / 5040.0 : 1.0 / 720.0);
            p = fma(p, z, odd ? -1.0 / 120.0 : -1.0 / 24.0);
            p = fma(p, z, odd ? 1.0 / 6.0 : 0.5);
        }
        const double W = (odd ? s3 : s2) * p;
        const double G2 = row_bc(W, 0), G3 = row_bc(W, 1);
        // even columns F = r0 s + qq G3 + u G2 - dt; odd G1 = s - beta G3 and r = T'(s) = r0 + u G1 + qq G2
        double Fr = fma(odd ? -beta : u, odd ? G3 : G2, odd ? s0 : -dt);
        const double G1 = row_bc(Fr, 1);
        Fr = fma(odd ? u : qq, odd ? Fr : G3, odd ? r0 : Fr);
        Fr = fma(odd ? qq : r0, odd ? G2 : s0, Fr);
        const double r = row_bc(Fr, 1);
        const F2 Fp = f2_split(row_bc(Fr, 0)), rp = f2_split(r);
        // Halley step dH = dN (1 - dN T''/(2 T')), dN = -F / r (a pair: dN is below 2^-20 s)
        const float ri = rcp_f32(rp.h);
        const F2 dN = f2_div(F2{-Fp.h, -Fp.l}, rp, ri);
        const float G2f = d2f_bits(G2), G1f = d2f_bits(G1), G0f = fmaf(-bf, G2f, 1.0f);
        const float kf = 0.5f * dN.h * fmaf(uf, G0f, qf * G1f) * ri;
        // G2(s + dH) = G2 + dH G1 (1 + dH G0 / (2 G1)), G3 + dH G2 (1 + dH G1 / (2 G2)); column 2: s + dH
        const float hf = 0.5f * dN.h * (odd ? G1f * rcp_f32(G2f) : G0f * rcp_f32(G1f));
        const double dl = f2_double(f2_norm(dN.h, fmaf(dN.h, (col == 2 ? 0.0f : hf) - kf, dN.l)));
        const double Gn = fma(dl, col == 2 ? 1.0 : (odd ? G2 : G1), col == 2 ? s0 : (odd ? G3 : G2));
        ok = ok && (__double2hiint(r) > 0) && fabsf(dN.h) <= 6.1035156e-5f * fabsf(sf);
        const double G2n = row_bc(Gn, 0), G3n = row_bc(Gn, 1);
        const double fg = fma(odd ? -mu : -mur0, odd ? G3n : G2n, odd ? dt : 0.0);  // f - 1, g
        const double fm1 = row_bc(fg, 0), g = row_bc(fg, 1);
        const double qc = own(q);
        wc = own(w);
        // rows without a planet stay where they are
        double qn = on ? fma(fm1, qc, fma(g, wc, qc)) : qc, wg = 0.0;
        if (__any_sync(kFullMask, on && !ok)) {
            // the general solver for the rows the fast path left
            if (on && !ok) {
                double a[3] = {q[0], q[1], q[2]}, b[3] = {w[0], w[1], w[2]};
                if (!drift_general(mu, dt, a[0], a[1], a[2], b[0], b[1], b[2])) failed = true;
                qn = own(a);
                wg = own(b);
            }
        }
        double qnew[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) qnew[d] = row_bc(qn, d);
        // |x|, mu/|x| of the new position; fdot, gdot - 1
        const double x2 = fma(qnew[0], qnew[0], fma(qnew[1], qnew[1], qnew[2] * qnew[2]));
        const double rinv = rsqrt_full(x2);
        const double G1n = fma(-beta, G3n, row_bc(Gn, 2));
        const double m1 = (col == 0 ? mur0 : (col == 1 ? mu : x2)) * rinv;
        const double m2 = -m1 * (col == 0 ? G1n : G2n);
        const double fd = row_bc(m2, 0), gdm1 = row_bc(m2, 1);
        const double wd = fma(fd, qc, fma(gdm1, wc, wc));
        wc = ok && on ? wd : wg;
        mur0 = row_bc(m1, 1);
        r0 = row_bc(m1, 2);
#pragma unroll
        for (int d = 0; d < 3; ++d) q[d] = qnew[d];
        eph_kick_any<H>(pc, ln, dt, q, r0, delta, K);
        // closing half kick: synchronised state at t_{k+1}
        wc = fma(0.5, K, wc);
        const int e = k + 1, b = e & 1;
        if (e >= 2) {
            eph_bar_sync(3 + b, threads);  // the other warps are done with emitted step e - 2
            if (__shfl_sync(kFullMask, *reinterpret_cast<volatile int*>(&ring.stop), 0)) {
                if (lane == 0) ring.last[b] = 1;
                __syncwarp();
                eph_bar_arrive(1 + b, threads);
                eph_bar_sync(3 + (b ^ 1), threads);
                return;
            }
        }
        eph_hand_over(ring, ln, b, qn, wc, delta, threads);
    }
    // wait for the other warps to finish the last emitted steps
    for (int e = nsteps > 0 ? nsteps - 1 : 0; e <= nsteps; ++e) eph_bar_sync(3 + (e & 1), threads);
    if (on && col < 3) {
        jac[3 * row + col] = own(q);
        jac[3 * np + 3 * row + col] = wc;
    }
    if (__any_sync(kFullMask, failed) && lane == 0) *status = GLISSE_E_KEPLER;
}

// Warps 1 and 2 of the block, for each emitted step e = 0..nsteps: warp 1 the log record
// (positions + h0, broadcast layout), warp 2 (blocks that keep a history) the synchronised
// heliocentric states hist[e][np][6].
// progress (optional, host-mapped): after every kProgressEvery-th step and the last, the
// number of steps whose entries are written, published with a system-scope fence so
// that the host may launch work on them while this runs.
// stop (optional): a word that another stream may set; seen, it ends the chunk early.
__device__ __forceinline__ void eph_emit(const PlanetConsts& pc, double dt, int nsteps, EphRing& ring,
                                         double* __restrict__ log, double* __restrict__ hist, int* progress,
                                         const int* stop, int threads) {
    const int np = pc.np;
    const int lane = threadIdx.x & 31;
    const bool writes_log = threadIdx.x < 64;
    const bool on = lane < np;
    const int S = log_stride(np);
    const double gm = on ? pc.gm[lane] : 0.0;
    const double m_over_eta = on ? pc.m[lane] / pc.eta[lane + 1] : 0.0;
    for (int e = 0; e <= nsteps; ++e) {
        const int b = e & 1;
        eph_bar_sync(1 + b, threads);
        if (*reinterpret_cast<volatile int*>(&ring.last[b])) break;
        double r[3], w[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            F2 del{0.0f, 0.0f};
            r[d] = on ? ring.q[b][lane][d] : 0.0;
            w[d] = on ? ring.w[b][lane][d] : 0.0;
            if (on) del = ring.d[b][lane][d];
            r[d] += f2_double(f2_norm(del.h, del.l));
        }
        if (writes_log && stop && (e % kStopEvery) == 0 && lane == 0 && *reinterpret_cast<const volatile int*>(stop))
            *reinterpret_cast<volatile int*>(&ring.stop) = 1;
        __syncwarp();
        eph_bar_arrive(3 + b, threads);  // the ring slot may be refilled
        if (writes_log) {
            // h0 = -sum_j G m_j r_j / |r_j|^3
            const double r2 = on ? fma(r[0], r[0], fma(r[1], r[1], r[2] * r[2])) : 1.0;
            const double own = -k_rcube(r2, gm);
            double h0[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                h0[d] = own * r[d];
                for (int o = 1; o < np; o <<= 1) h0[d] += __shfl_xor_sync(kFullMask, h0[d], o);
            }
            double* L = log + (size_t)e * S;
            if (on) store_rec(L + kRec * lane, r[0], r[1], r[2], r[0], r[1], r[2]);
            if (lane == 0) store_rec(L + kRec * np, h0[0], h0[1], h0[2], dt * h0[0], dt * h0[1], dt * h0[2]);
        } else {
            double* Hs = hist + (size_t)e * 6 * np;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double vh = w[d] + warp_excl_prefix(m_over_eta * w[d], lane, np);
                if (on) {
                    Hs[6 * lane + d] = r[d];
                    Hs[6 * lane + 3 + d] = vh;
                }
            }
        }
        if (progress && e > 0 && ((e % kProgressEvery) == 0 || e == nsteps)) {
            __threadfence_system();  // every lane's entries before the count
            if (hist) eph_bar_sync(5, 64);
            __syncwarp();
            if (writes_log && lane == 0) *reinterpret_cast<volatile int*>(progress) = e;
        }
    }
}

constexpr int kEphThreads = 96;        // warps 0 to 2
constexpr int kEphThreadsNoHist = 64;  // no history: warps 0 and 1

// The block's threads are kEphThreads with a history, else kEphThreadsNoHist.
__device__ __forceinline__ void eph_advance(const PlanetConsts& pc, double* jac, double dt, int nsteps,
                                            double* __restrict__ log, double* __restrict__ hist, int* status,
                                            int* progress = nullptr, const int* stop = nullptr) {
    __shared__ EphRing ring;
    const int threads = hist ? kEphThreads : kEphThreadsNoHist;
    if (threadIdx.x == 0) ring.stop = ring.last[0] = ring.last[1] = 0;
    __syncthreads();
    if (threadIdx.x < 32) {
        if (pc.np > kEphCols)
            eph_dynamics<2>(pc, jac, dt, nsteps, ring, status, threads);
        else
            eph_dynamics<1>(pc, jac, dt, nsteps, ring, status, threads);
    } else {
        eph_emit(pc, dt, nsteps, ring, log, hist, progress, stop, threads);
    }
}

__global__ void __launch_bounds__(kEphThreads) eph_chunk_kernel(const PlanetConsts* __restrict__ pcp, double* jac,
                                                                  double dt, int nsteps, double* __restrict__ log,
                                                                  double* __restrict__ hist, int* status,
                                                                  int* progress, const int* stop) {
    eph_advance(*pcp, jac, dt, nsteps, log, hist, status, progress, stop);
}

// Many independent systems: block b advances system b.
//   jac  : [n_sys][2][kMaxPlanets][3] Jacobi states (per-system stride 6 kMaxPlanets)
//   log  : system b's log at log + log_off[b] (stride log_stride(np_b) doubles per step)
//   dt   : [n_sys] steps
__global__ void __launch_bounds__(kEphThreadsNoHist) eph_batch_kernel(const PlanetConsts* __restrict__ pcs, double* jac,
                                                                        const double* __restrict__ dt, int nsteps,
                                                                        double* __restrict__ log,
                                                                        const int64_t* __restrict__ log_off,
                                                                        int* status) {
    const int b = blockIdx.x;
    eph_advance(pcs[b], jac + (size_t)b * 6 * kMaxPlanets, dt[b], nsteps, log + log_off[b], nullptr, status);
}

// ---------------------------------------------------------------------------
// External positions -> log layout with h0.  One thread per step.
//   pos : [n+1][np][3] heliocentric positions
// ---------------------------------------------------------------------------
__global__ void eph_external_kernel(const PlanetConsts* __restrict__ pcp, const double* __restrict__ pos, int64_t n1,
                                    double dt, double* __restrict__ log) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n1) return;
    const int np = pcp->np;
    const int S = log_stride(np);
    double hx = 0.0, hy = 0.0, hz = 0.0;
    for (int j = 0; j < np; ++j) {
        const double x = pos[(k * np + j) * 3 + 0], y = pos[(k * np + j) * 3 + 1], z = pos[(k * np + j) * 3 + 2];
        const double r2 = fma(x, x, fma(y, y, z * z));
        const double s = k_rcube(r2, pcp->gm[j]);
        hx = fma(-s, x, hx);
        hy = fma(-s, y, hy);
        hz = fma(-s, z, hz);
        store_rec(log + k * S + kRec * j, x, y, z, x, y, z);
    }
    store_rec(log + k * S + kRec * np, hx, hy, hz, dt * hx, dt * hy, dt * hz);
}

// host launchers ----------------------------------------------------------------
cudaError_t launch_eph_setup(const double* planets, int np, double m0, double G, int enc_mode, double enc_value,
                             PlanetConsts* pc, double* jac, int* status, cudaStream_t s) {
    eph_setup_kernel<<<1, 32, 0, s>>>(planets, np, m0, G, enc_mode, enc_value, pc, jac, status);
    return cudaGetLastError();
}

// The ephemeris is one serial block of two warps.  Sharing an SM partition
// with particle warps would slow it by the number of warps it shares the FP64
// pipe with, so its block asks for the largest dynamic shared-memory
// allocation a block may have: no other block fits on that SM while it runs
// (the memory is unused).  The particle grids are sized for the other SMs.
// In steady state the planets run a chunk ahead and the reservation changes
// nothing measurable (the step time agreed to 0.01% without it); it matters
// in the first chunk of a context, where the particles follow the planets a
// few steps behind and a slowed ephemeris would hold them back.
cudaError_t launch_eph_chunk(const PlanetConsts* pc, double* jac, double dt, int nsteps, double* log, double* hist,
                             int* status, cudaStream_t s, int* progress, const int* stop) {
    int dev = 0, optin = 0;
    cudaFuncAttributes fa{};
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, eph_chunk_kernel);
    // all of a block's shared memory: the kernel's own hand-off ring plus the rest as dynamic
    const int dyn = optin - (int)fa.sharedSizeBytes;
    if (e == cudaSuccess && dyn < 0) e = cudaErrorInvalidConfiguration;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(eph_chunk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    if (e != cudaSuccess) return e;
    eph_chunk_kernel<<<1, hist ? kEphThreads : kEphThreadsNoHist, (size_t)dyn, s>>>(pc, jac, dt, nsteps, log, hist,
                                                                                    status, progress, stop);
    return cudaGetLastError();
}

cudaError_t launch_eph_batch(const PlanetConsts* pcs, int n_sys, double* jac, const double* dt, int nsteps,
                             double* log, const int64_t* log_off, int* status, cudaStream_t s) {
    if (n_sys <= 0) return cudaSuccess;
    eph_batch_kernel<<<n_sys, kEphThreadsNoHist, 0, s>>>(pcs, jac, dt, nsteps, log, log_off, status);
    return cudaGetLastError();
}

cudaError_t launch_eph_external(const PlanetConsts* pc, const double* pos, int64_t n1, double dt, double* log,
                                cudaStream_t s) {
    const int bs = 128;
    const int64_t grid = (n1 + bs - 1) / bs;
    eph_external_kernel<<<(unsigned)grid, bs, 0, s>>>(pc, pos, n1, dt, log);
    return cudaGetLastError();
}

}  // namespace glisse
