// particle_map.cuh -- the test-particle map over one segment of a planet chunk
// (shared by the translation units that instantiate it for each drift mode).
//
// Section 2.2: one thread per particle; the particle is loaded once, carried
// in registers through every step of the chunk, and stored once.  Each step
// is kick(dt/2) - Kepler drift(dt) - kick(dt/2) with the kick
//   dv/dt = h0 - sum_j G m_j (r - r_j) / |r - r_j|^3,  h0 = -sum_j G m_j r_j / |r_j|^3,
// and the removal test (encounter |r - r_j| < R_crit,j, escape |r| > r_max)
// made at every kick time on the drifted position.  Inside a segment the
// closing half kick of step k and the opening half kick of step k+1 use the
// same planet positions, so they are applied as one kick of dt.  A context's
// segments end "open": the last step ends with the same full kick that an
// uncut launch would apply there, the stored velocities already carry the
// next step's opening half kick, and the next segment skips it (open_in /
// close_out = 0).  Cuts then leave no trace: any split of a run into calls,
// pieces or sample stops gives the same bits.  The synchronised state the
// caller reads (velocities with only the closing half kick) is computed at
// the cut by one extra half kick from the same pre-kick velocities and
// written by id (publish).  close_out = 1 ends with the closing half kick
// instead, leaving the synchronised state in the slots (batched systems).
//
// The batched kernel may hold one particle in a lane pair (TPP = 2): both
// lanes run the same state and drift, each takes half of the planets in the
// kick, and the pair adds its two partial kicks (kick_test_pair).
//
// A removed particle keeps the state it had after the drift and before the
// closing kick, gets removal_step = k+1 and the reason (planet 1..N_p, lowest
// index first; encounter before escape), and its lane idles until the warp
// finishes or compaction drops it.  A failed Kepler solve or a non-finite
// result keeps the state from before the drift (reasons -2 / -3).
#pragma once
#include <algorithm>
#include "glisse_internal.h"
#include "kepler.cuh"
#include "split_step.cuh"

namespace glisse {

constexpr int kParticleBlock = 128;
// Resident blocks per SM the particle kernel is compiled for (register budget
// 65536 / (128 x blocks)).  A chunk's warps all do the same work, so a launch
// that spills past one wave leaves a tail in which a lone warp per SM
// partition cannot keep the FP64 pipe busy.
#ifndef GLISSE_PARTICLE_MIN_BLOCKS
#define GLISSE_PARTICLE_MIN_BLOCKS 4
#endif

// drift used by the particle map: the converged fast solver (default) or the
// paper's fixed-iteration solve (GLISSE_KEPLER_PAPER_FIXED)
constexpr int kDriftConverge = 0;
constexpr int kDriftPaper = 1;
constexpr int kAnyNp = -1;  // planet count at run time

// Read-only broadcast loads of one log record: its doubles, and its pairs.
__device__ __forceinline__ void load_rec(const double* __restrict__ p, double& x, double& y, double& z) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p));
    x = a.x;
    y = a.y;
    z = __ldg(p + 2);
}

__device__ __forceinline__ void load_rec_split(const double* __restrict__ p, F2 (&v)[3]) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p + kRecSplit));
    const float2 b = __ldg(reinterpret_cast<const float2*>(p + kRecSplit + 2));
    v[0] = F2{a.x, a.w};
    v[1] = F2{a.y, b.x};
    v[2] = F2{a.z, b.y};
}

// The terms that kick_sum leaves to FP64 (bit j of `near`: planet j, bit np: h0), for
// one lane: added to K, with the encounter test.  Returns the lowest 1-based
// planet index whose test fires, or 0.
__device__ __forceinline__ int kick_near(unsigned near, int np, double x, double y, double z,
                                         const double* __restrict__ L, const ParticleConsts& pc, double (&K)[3]) {
    int hit = 0;
    if ((near >> np) & 1u) {
        double hx, hy, hz;
        load_rec(L + kRec * np, hx, hy, hz);
        K[0] = fma(pc.dt, hx, K[0]);
        K[1] = fma(pc.dt, hy, K[1]);
        K[2] = fma(pc.dt, hz, K[2]);
    }
#pragma unroll 1
    for (int j = np - 1; j >= 0; --j) {
        if (!((near >> j) & 1u)) continue;
        double px, py, pz;
        load_rec(L + kRec * j, px, py, pz);
        const double dx = x - px, dy = y - py, dz = z - pz;
        const double d2 = fma(dx, dx, fma(dy, dy, dz * dz));
        hit = lt_nonneg(d2, pc.rc2[j]) ? (j + 1) : hit;
        const double s = k_rcube(d2, pc.tgm_full[j]);
        K[0] = fma(-s, dx, K[0]);
        K[1] = fma(-s, dy, K[1]);
        K[2] = fma(-s, dz, K[2]);
    }
    return hit;
}

// The kick of a full step, K = dt a(r) at log step L (a half kick is exactly half
// of it), and the encounter test: h0 and the planets in pairs (kick_split), in
// FP64 (N) the planets a lane is near to, and the whole sum where it exceeds 2^-7 |v|
// (far out, where h0 outweighs the star: a pair's 46 bits of K would show in v).
// base: the part of the drift's velocity still in pairs; on return C = base + K - N.
// X: the position split; sp.v2 is negative where the position is out of the
// floats' range (then all is FP64).  Returns the lowest 1-based planet index whose
// test fires, or 0; *exact: some lane's N is not zero.  All lanes of a warp call it
// together.
// TPP = 2: a lane pair (both lanes holding the same particle) splits the planets:
// lane parity p takes planets p, p + 2, ..., the partial sums are added (the
// same bits on both lanes: two_sum and addition commute) and the lower index wins.
// NP: the planet count, or kAnyNp to take it from np_any (one code for all counts, a rolled
// loop: in kernels with much code the shorter loop is the faster one, 23.2 against 24.6 ms
// for the batch's chunk unrolled by two; the unrolled one is for the single-system
// kernels, 6.5 against 6.9 ms for 131072 particles).
// WARP false: one lane by itself (*exact is the lane's own).
template <int NP, int TPP, bool WARP = true>
__device__ __forceinline__ int kick_sum(int np_any, double x, double y, double z, const F2 (&X)[3],
                                        const F2 (&base)[3], const Speed& sp, bool act, const double* __restrict__ L,
                                        const ParticleConsts& pc, const SplitConsts& sc, F2 (&C)[3], double (&N)[3],
                                        bool& exact) {
    const int np = NP >= 0 ? NP : np_any;
    constexpr int kUnroll = NP >= 0 ? kMaxPlanets : 1;
    const int parity = TPP == 2 ? (int)(threadIdx.x & 1) : 0;
    const float lim2 = kSplitNear2 * sp.rate2;
    load_rec_split(L + kRec * np, C);
#pragma unroll
    for (int c = 0; c < 3; ++c) C[c] = TPP == 2 && parity == 1 ? F2{0.0f, 0.0f} : f2_add(base[c], C[c]);
    unsigned near = 0, mine = parity == 0 ? 1u << np : 0u;
#pragma unroll kUnroll
    for (int jj = (np + TPP - 1) / TPP - 1; jj >= 0; --jj) {
        const int j = TPP * jj + parity;
        if (j < np) {
            F2 P[3];
            load_rec_split(L + kRec * j, P);
            if (!kick_split(X, P, sc.tg[j], sc.rc2[j], lim2, C)) near |= 1u << j;
            mine |= 1u << j;
        }
    }
    if constexpr (TPP == 2) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            C[c] = f2_add(C[c], F2{__shfl_xor_sync(kFullMask, C[c].h, 1), __shfl_xor_sync(kFullMask, C[c].l, 1)});
    }
    const float k2 = fmaf(C[0].h, C[0].h, fmaf(C[1].h, C[1].h, C[2].h * C[2].h));
    const bool small = k2 <= kSplitKick2 * sp.v2;
    int hit = 0;
    exact = act && (near != 0u || !small);
    if constexpr (WARP) exact = __any_sync(kFullMask, exact);
    if (exact) {
        N[0] = N[1] = N[2] = 0.0;
        if (!small) {
            near = mine;
#pragma unroll
            for (int c = 0; c < 3; ++c) C[c] = base[c];
        }
        if (!act) near = 0;
        if (TPP == 2 || near) hit = kick_near(near, np, x, y, z, L, pc, N);
        if constexpr (TPP == 2) {
#pragma unroll
            for (int c = 0; c < 3; ++c) N[c] += __shfl_xor_sync(kFullMask, N[c], 1);
            const int other = __shfl_xor_sync(kFullMask, hit, 1);
            hit = (hit != 0 && other != 0) ? min(hit, other) : (hit | other);
        }
    }
    return hit;
}

__device__ __forceinline__ double f2_sum(const F2& v) { return f2_double(f2_norm(v.h, v.l)); }

// The FP64 drift (kepler.cuh) of the lanes that the pairs leave (part): the fast
// path, then the general solver for lanes outside its domain.  Returns false for a
// lane whose solve failed.  All lanes of a warp call it together.
static __device__ __noinline__ bool drift_fp64(const ParticleConsts& pc, bool part, double (&s)[6]) {
    double r0, mur0;
    radius_of(s[0], s[1], s[2], r0, mur0);
    mur0 *= pc.mu;
    const bool done = drift_fast(pc.mu, d2f_bits(pc.mu), pc.dt, d2f_bits(pc.dt), part, r0, mur0, s[0], s[1], s[2],
                                 s[3], s[4], s[5]);
    if (part && !done) return drift_general(pc.mu, pc.dt, s[0], s[1], s[2], s[3], s[4], s[5]);
    return true;
}

// Removal test without a kick (used at t_0).
__device__ __forceinline__ int test_only(int np, double x, double y, double z, const double* __restrict__ L,
                                         const double (&rc2)[kMaxPlanets], double rmax2) {
    int hit = 0;
    const double r2 = fma(x, x, fma(y, y, z * z));
    if (__double_as_longlong(rmax2) != 0 && lt_nonneg(rmax2, r2)) hit = GLISSE_REMOVED_ESCAPE;
#pragma unroll 1
    for (int j = np - 1; j >= 0; --j) {
        double px, py, pz;
        load_rec(L + kRec * j, px, py, pz);
        const double dx = x - px, dy = y - py, dz = z - pz;
        const double d2 = fma(dx, dx, fma(dy, dy, dz * dz));
        hit = lt_nonneg(d2, rc2[j]) ? (j + 1) : hit;
    }
    return hit;
}

// The map for one lane over nsteps steps of the log L (L step 0 = the lane's
// current time).  State in registers; act / reason / rstep record removal.
// open_in: the velocities already carry the opening half kick of step 0.
// close_out: false leaves the state open, ending with the full kick that a
// single longer launch would apply there (the next segment then has open_in).
// A split with open_in / close_out is bit-identical to no split.
// pc may live in the constant bank (kernel parameter) or in shared memory.
// TPP = 2: the particle is held by a lane pair (batched kernel), each lane
// running the same state with half of the planets in the kicks.
// Where a lane publishes its synchronised state: out[6 id[slot] .. + 5] (out null: nowhere).
struct PublishTo {
    const int32_t* id;
    double* out;
    int64_t slot;
};

// PUBLISH (with close_out false): a lane still live at the segment's end also
// writes its synchronised state there (position; pre-kick velocities plus the
// closing half kick), straight to memory so that nothing stays live in
// registers across the steps.
template <int NP, int MODE = kDriftConverge, int TPP = 1, bool PUBLISH = false>
__device__ __forceinline__ void advance_lane(const ParticleConsts& pc, const SplitConsts& sc,
                                             const double* __restrict__ L, int64_t step0, int nsteps, bool test_first,
                                             double& x, double& y, double& z, double& vx, double& vy, double& vz,
                                             bool& act, int& reason, int64_t& rstep, bool open_in = false,
                                             bool close_out = true, PublishTo pub = {}, int np_any = 0) {
    const int np = NP >= 0 ? NP : np_any;
    const int S = log_stride(np);

    if (test_first) {
        const int h = test_only(np, x, y, z, L, pc.rc2, pc.rmax2);
        if (act && h != 0) {
            act = false;
            reason = h;
            rstep = step0;
        }
    }
    F2 X[3] = {f2_split(x), f2_split(y), f2_split(z)};
    double r2 = fma(x, x, fma(y, y, z * z));
    constexpr F2 kZero = {0.0f, 0.0f};
    if (!open_in) {
        const F2 base[3] = {kZero, kZero, kZero};
        F2 C[3];
        double N[3];
        bool exact;
        kick_sum<NP, TPP>(np, x, y, z, X, base, float_speed(r2, vx, vy, vz), act, L, pc, sc, C, N, exact);
        if (act) {
            vx = fma(0.5, f2_sum(C[0]), vx);
            vy = fma(0.5, f2_sum(C[1]), vy);
            vz = fma(0.5, f2_sum(C[2]), vz);
            if (exact) {
                vx = fma(0.5, N[0], vx);
                vy = fma(0.5, N[1], vy);
                vz = fma(0.5, N[2], vz);
            }
        }
    }

    bool all_slow = false;
    for (int k = 0; k < nsteps; ++k) {
        if (!__any_sync(kFullMask, act)) break;
        const double* __restrict__ Ln = L + (size_t)(k + 1) * S;
        // the drifted position n[0..2] and velocity n[3..5] + base: (gdot - 1) v stays in pairs,
        // to enter the velocity in one sum with the kick
        double n[6];
        F2 base[3] = {kZero, kZero, kZero};
        bool failed = false;
        Speed sp;
        if constexpr (MODE == kDriftConverge) {
            const F2 V[3] = {f2_split(vx), f2_split(vy), f2_split(vz)};
            DriftFactors f = {0.0, 0.0, 0.0, kZero};
            bool slow = act;
            // a warp whose lanes all stepped too far for the pairs spares itself the attempt while
            // m alone says so (same results: those lanes take the FP64 drift either way)
            if (!all_slow || __any_sync(kFullMask, act && !beyond_split(r2, d2f_bits(sc.mudt), sc.dt.h)))
                slow = !drift_split(r2, sc.mudt, pc.dt, sc.dt, X, V, f, sp) && act;
            else
                sp = split_speed(r2, sc.mudt, V);
#pragma unroll
            for (int c = 0; c < 3; ++c) base[c] = f2_mul(f.gdm1, V[c]);
            n[0] = fma(f.fm1, x, fma(f.g, vx, x));
            n[1] = fma(f.fm1, y, fma(f.g, vy, y));
            n[2] = fma(f.fm1, z, fma(f.g, vz, z));
            n[3] = fma(f.fd, x, vx);
            n[4] = fma(f.fd, y, vy);
            n[5] = fma(f.fd, z, vz);
            if (__any_sync(kFullMask, slow)) {
                double s[6] = {x, y, z, vx, vy, vz};
                all_slow = __all_sync(kFullMask, slow || !act);
                const bool done = drift_fp64(pc, slow, s);
                if (slow) {
                    failed = !done;
#pragma unroll
                    for (int c = 0; c < 6; ++c) n[c] = s[c];
                    base[0] = base[1] = base[2] = kZero;
                }
            }
        } else {
            sp = float_speed(r2, vx, vy, vz);
            n[0] = x;
            n[1] = y;
            n[2] = z;
            n[3] = vx;
            n[4] = vy;
            n[5] = vz;
            if (act)
                failed = drift_paper(pc.mu, pc.dt, pc.kepler_iters, pc.kepler_tol, n[0], n[1], n[2], n[3], n[4],
                                     n[5]) != 0;
        }
        const bool bad = nonfinite_bits(n[0]) || nonfinite_bits(n[1]) || nonfinite_bits(n[2]) ||
                         nonfinite_bits(n[3]) || nonfinite_bits(n[4]) || nonfinite_bits(n[5]);
        if (act && (failed || bad)) {
            // the state stays what it was before the drift
            act = false;
            reason = failed ? GLISSE_REMOVED_KEPLER : GLISSE_REMOVED_NONFINITE;
            rstep = step0 + k + 1;
        }
        if (act) {
            x = n[0];
            y = n[1];
            z = n[2];
            vx = n[3];
            vy = n[4];
            vz = n[5];
        }
        X[0] = f2_split(x);
        X[1] = f2_split(y);
        X[2] = f2_split(z);
        r2 = fma(x, x, fma(y, y, z * z));
        // escape: |r|^2 > r_max^2 (integer compare of non-negative doubles)
        int hit = (__double_as_longlong(pc.rmax2) != 0 && lt_nonneg(pc.rmax2, r2)) ? GLISSE_REMOVED_ESCAPE : 0;
        if (!in_float_range(r2)) sp.v2 = -1.0f;
        F2 C[3];
        double N[3];
        bool exact;
        const int enc = kick_sum<NP, TPP>(np, x, y, z, X, base, sp, act, Ln, pc, sc, C, N, exact);
        hit = enc ? enc : hit;
        const bool last = k + 1 == nsteps;
        if (last) {
            // the synchronised state: drift and half of the kick, base + K/2 = (base + C) / 2
            if (act && hit == 0 && (close_out || (PUBLISH && pub.out))) {
                double h[3] = {vx, vy, vz};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    h[c] = fma(0.5, f2_sum(f2_add(base[c], C[c])), h[c]);
                    if (exact) h[c] = fma(0.5, N[c], h[c]);
                }
                if (close_out) {
                    vx = h[0];
                    vy = h[1];
                    vz = h[2];
                    break;
                }
                if constexpr (PUBLISH) {
                    double* o = pub.out + 6 * (int64_t)pub.id[pub.slot];
                    o[0] = x;
                    o[1] = y;
                    o[2] = z;
                    o[3] = h[0];
                    o[4] = h[1];
                    o[5] = h[2];
                }
            }
        }
        if (act) {
            // a removed particle keeps the drifted velocity
            if (hit != 0) {
                act = false;
                reason = hit;
                rstep = step0 + k + 1;
#pragma unroll
                for (int c = 0; c < 3; ++c) C[c] = base[c];
            }
            vx += f2_sum(C[0]);
            vy += f2_sum(C[1]);
            vz += f2_sum(C[2]);
            if (exact && act) {
                vx += N[0];
                vy += N[1];
                vz += N[2];
            }
        }
    }
}

// Write a removed particle's result under its id.
__device__ __forceinline__ void store_removed(int64_t pid, double x, double y, double z, double vx, double vy,
                                              double vz, int64_t rstep, int reason, double* out_state,
                                              int64_t* out_step, int32_t* out_reason) {
    double* o = out_state + 6 * pid;
    o[0] = x;
    o[1] = y;
    o[2] = z;
    o[3] = vx;
    o[4] = vy;
    o[5] = vz;
    out_step[pid] = rstep;
    out_reason[pid] = reason;
}

template <int NP, int MODE>
__global__ void __launch_bounds__(kParticleBlock, GLISSE_PARTICLE_MIN_BLOCKS)
    particle_chunk_kernel(const ChunkArgs a, const __grid_constant__ ParticleConsts pc,
                          const __grid_constant__ SplitConsts sc) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool in = i < a.n;
    const int64_t ld = a.ld;
    double x, y, z, vx, vy, vz;
    if (in) {
        x = a.st[i];
        y = a.st[ld + i];
        z = a.st[2 * ld + i];
        vx = a.st[3 * ld + i];
        vy = a.st[4 * ld + i];
        vz = a.st[5 * ld + i];
    } else {
        // idle lanes carry a harmless circular orbit so the shared drift stays finite
        x = 1.0;
        y = 0.0;
        z = 0.0;
        vx = 0.0;
        vy = 6.283185307179586;
        vz = 0.0;
    }
    bool act = in && a.alive[i] != 0;
    const bool started = act;
    int reason = 0;
    int64_t rstep = -1;
    advance_lane<NP, MODE, 1, true>(pc, sc, a.log, a.step0, a.nsteps, a.test_first != 0, x, y, z, vx, vy, vz, act,
                                    reason, rstep, a.open_in != 0, a.close_out != 0, PublishTo{a.id, a.out_state, i});
    if (a.steps_done) {
        // steps this particle actually advanced in the segment (exact work count)
        const unsigned adv = !started ? 0u : (rstep >= 0 ? (unsigned)(rstep - a.step0) : (unsigned)a.nsteps);
        const unsigned wsum = __reduce_add_sync(kFullMask, adv);
        if ((threadIdx.x & 31) == 0 && wsum) atomicAdd(a.steps_done, (unsigned long long)wsum);
    }
    if (a.live_out) {
        // particles live at the segment's end
        const unsigned wl = __reduce_add_sync(kFullMask, act ? 1u : 0u);
        if ((threadIdx.x & 31) == 0 && wl) atomicAdd(a.live_out, (unsigned long long)wl);
    }
    if (in) {
        a.st[i] = x;
        a.st[ld + i] = y;
        a.st[2 * ld + i] = z;
        a.st[3 * ld + i] = vx;
        a.st[4 * ld + i] = vy;
        a.st[5 * ld + i] = vz;
        a.alive[i] = act ? 1 : 0;
        if (rstep >= 0) store_removed(a.id[i], x, y, z, vx, vy, vz, rstep, reason, a.out_state, a.out_step,
                                      a.out_reason);
    }
}

// ---------------------------------------------------------------------------
// Task mode: persistent warps over (group, sub-chunk) tasks.
//
// With one thread per slot a chunk lasts as long as the SM partition holding the
// most warps, or the slowest ones (a group with a particle near a planet or a
// pericentre takes longer).  A particle's steps are serial, so balance needs
// smaller units of work: the segment is cut into sub-chunks of sub_steps steps, and
// a task is one group of 32 slots (the members of one warp of the plain launch) over
// one sub-chunk.  A fixed number of resident warps takes tasks: the first sub-chunk
// of every group in order, then whichever group's previous sub-chunk finished
// first (a queue: a finished task appends its group's next one).  With more groups
// than resident warps a task is nearly always ready.  A group that has fallen behind
// the others (one with a particle near a planet or a pericentre) is not put back:
// its warp goes on with it, so that it does not finish last.  Sub-chunk cuts are
// open cuts, so the result is bit-identical to the plain launch: same members per warp,
// same steps, same kicks.
//
// A warp without a task waits, bounded, until its entry of the queue appears or every
// group is finished.  The wait cannot deadlock: an unfinished group is either being
// run (and its task ends in an append, in the next task or in the group's end) or in the
// queue; if every running warp waited, all tickets before the first waiting one
// would have been used up, the unfinished groups would be appended entries that no
// ticket took, and the first waiting ticket is the next of those.
// ---------------------------------------------------------------------------
constexpr int kSubSteps = 32;
constexpr int kMaxSub = 32;  // sub-chunks per segment at most (5 bits of a queue entry)
// a wait for the queue gives up after this many polls (~64 ns each: seconds, where a
// sub-chunk takes a millisecond at most)
constexpr int kGroupWaitPolls = 1 << 25;

__host__ __device__ inline int task_sub_steps(int nsteps) {
    return max(kSubSteps, (nsteps + kMaxSub - 1) / kMaxSub);
}

__device__ __forceinline__ unsigned ld_acquire(const uint32_t* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(uint32_t* p, unsigned v) {
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// queue[0] counts the appends, queue[1] the finished groups; queue[2 + k] is the k-th append:
// 1 + 32 group + sub-chunk.
enum TaskState { kTaskReady, kTaskNone, kTaskTimeout };

// The task of ticket t: group and sub-chunk (the same on the whole warp).
__device__ __forceinline__ TaskState task_of_ticket(int64_t t, int64_t n_groups, const uint32_t* queue,
                                                    int polls_limit, int64_t& g, int& s) {
    if (t < n_groups) {
        g = t;
        s = 0;
        return kTaskReady;
    }
    unsigned v = 0;
    int state = kTaskReady;
    if ((threadIdx.x & 31) == 0) {
        const int limit = polls_limit > 0 ? polls_limit : kGroupWaitPolls;
        const uint32_t* p = queue + 2 + (t - n_groups);
        int polls = 0;
        while ((v = ld_acquire(p)) == 0u) {
            if ((int64_t)ld_acquire(queue + 1) >= n_groups) {
                state = kTaskNone;
                break;
            }
            if (++polls >= limit) {
                state = kTaskTimeout;
                break;
            }
            __nanosleep(64);
        }
    }
    v = __shfl_sync(kFullMask, v, 0);
    state = __shfl_sync(kFullMask, state, 0);
    __syncwarp();
    g = (int64_t)((v - 1u) >> 5);
    s = (int)((v - 1u) & 31u);
    return (TaskState)state;
}

// After task (g, s): publishes every lane's stores.  True when the warp is to go on with
// (g, s + 1): the group is behind by more than half of the tasks that the queue holds
// (warps: resident warps; taken: the ticket counter).  Else the group's next task goes
// to the queue, or the group is finished.
template <class Counter>
__device__ __forceinline__ bool task_done(uint32_t* queue, const Counter* taken, int64_t g, int s, int n_sub,
                                          int64_t n_groups, int64_t warps) {
    __threadfence();
    __syncwarp();
    int on = 0;
    if ((threadIdx.x & 31) == 0) {
        if (s + 1 >= n_sub) {
            if (n_sub > 1) atomicAdd(queue + 1, 1u);
        } else {
            const int64_t now = (int64_t)*reinterpret_cast<const volatile Counter*>(taken);
            on = 2 * (now - (s * n_groups + g)) > n_groups + warps;
            if (!on) {
                const unsigned pos = atomicAdd(queue, 1u);
                st_release(queue + 2 + pos, 1u + 32u * (unsigned)g + (unsigned)(s + 1));
            }
        }
    }
    return __shfl_sync(kFullMask, on, 0) != 0;
}

// at most five blocks per SM (task_warps_per_partition), so up to 96 registers per thread
constexpr int kTaskMaxBlocks = 5;

template <int NP>
__global__ void __launch_bounds__(kParticleBlock, kTaskMaxBlocks)
    particle_tasks_kernel(const ChunkArgs a, const __grid_constant__ ParticleConsts pc,
                          const __grid_constant__ SplitConsts sc, const TaskArgs ta) {
    const int lane = threadIdx.x & 31;
    const int64_t ld = a.ld;
    const int S = log_stride(NP);
    const int n_sub = (a.nsteps + ta.sub_steps - 1) / ta.sub_steps;
    const int64_t n_tasks = (int64_t)ta.n_groups * n_sub;
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(ta.task_counter, 1ull);
        t = __shfl_sync(kFullMask, t, 0);
        if ((int64_t)t >= n_tasks) break;
        int64_t g;
        int s;
        const TaskState got = task_of_ticket((int64_t)t, ta.n_groups, ta.queue, ta.wait_polls, g, s);
        if (got == kTaskTimeout && lane == 0) atomicExch(ta.status, GLISSE_E_TIMEOUT);
        if (got != kTaskReady) break;
        do {
            const int64_t i = g * 32 + lane;
            const bool in = i < a.n;
            double x = 1.0, y = 0.0, z = 0.0, vx = 0.0, vy = 6.283185307179586, vz = 0.0;
            bool act = false;
            if (in) {
                // written by another warp's task (L2 is coherent, this SM's L1 may not be)
                x = __ldcg(a.st + i);
                y = __ldcg(a.st + ld + i);
                z = __ldcg(a.st + 2 * ld + i);
                vx = __ldcg(a.st + 3 * ld + i);
                vy = __ldcg(a.st + 4 * ld + i);
                vz = __ldcg(a.st + 5 * ld + i);
                act = __ldcg(a.alive + i) != 0;
            }
            const bool started = act;
            int reason = 0;
            int64_t rstep = -1;
            const int k0 = s * ta.sub_steps;
            const int m = min(ta.sub_steps, a.nsteps - k0);
            const bool last = s + 1 == n_sub;
            advance_lane<NP, kDriftConverge, 1, true>(pc, sc, a.log + (size_t)k0 * S, a.step0 + k0, m,
                                                      a.test_first != 0 && s == 0, x, y, z, vx, vy, vz, act, reason,
                                                      rstep, s > 0 || a.open_in != 0, last ? a.close_out != 0 : false,
                                                      PublishTo{a.id, last ? a.out_state : nullptr, i});
            if (a.steps_done) {
                const unsigned adv = !started ? 0u : (rstep >= 0 ? (unsigned)(rstep - (a.step0 + k0)) : (unsigned)m);
                const unsigned wsum = __reduce_add_sync(kFullMask, adv);
                if (lane == 0 && wsum) atomicAdd(a.steps_done, (unsigned long long)wsum);
            }
            if (last && a.live_out) {
                const unsigned wl = __reduce_add_sync(kFullMask, act ? 1u : 0u);
                if (lane == 0 && wl) atomicAdd(a.live_out, (unsigned long long)wl);
            }
            if (in) {
                __stcg(a.st + i, x);
                __stcg(a.st + ld + i, y);
                __stcg(a.st + 2 * ld + i, z);
                __stcg(a.st + 3 * ld + i, vx);
                __stcg(a.st + 4 * ld + i, vy);
                __stcg(a.st + 5 * ld + i, vz);
                __stcg(a.alive + i, (uint8_t)(act ? 1 : 0));
                if (rstep >= 0) store_removed(a.id[i], x, y, z, vx, vy, vz, rstep, reason, a.out_state, a.out_step,
                                              a.out_reason);
            }
        } while (task_done(ta.queue, ta.task_counter, g, s++, n_sub, ta.n_groups,
                           (int64_t)gridDim.x * (kParticleBlock / 32)));
    }
}

// Dynamic shared memory (unused by the kernel) that caps the resident blocks
// per SM at what an even spread of this grid needs.  Every block does the same
// work, so the chunk lasts as long as the SM holding the most blocks; the
// hardware may pack up to GLISSE_PARTICLE_MIN_BLOCKS on some SMs and fewer on
// others, and the ephemeris kernel holds one SM for itself (all of its shared
// memory).  Spread over the other SMs, ceil(grid / (SMs - 1)) per SM is the
// best any placement can do; the request makes more than that impossible.
inline cudaError_t particle_smem_cap(const void* kernel, int64_t grid, size_t* smem) {
    *smem = 0;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t per_sm = nsm > 1 ? (grid + nsm - 2) / (nsm - 1) : GLISSE_PARTICLE_MIN_BLOCKS;
    return residency_cap_smem(kernel, per_sm, GLISSE_PARTICLE_MIN_BLOCKS, smem);
}

// Warps per SM partition for task mode, or 0 for the plain launch.  Few warps leave the
// FP64 pipe idle between a warp's dependent instructions; many make a group's
// sub-chunks slower, and with it the tail in which the last groups finish.  Milliseconds
// per 1024 steps at 2 | 3 | 4 | 5 warps (8 bodies, particles at 2-46 au, groups per partition in
// brackets; plain launch in front):
//     32768 [1.7]   2.8: 2.9 | 3.1 | 3.5 | 4.8        65536 [3.4]   4.5: 4.3 | 4.0 | 4.3 | 4.5
//     98304 [5.1]   6.9: 6.3 | 5.3 | 5.4 | 5.6       131072 [6.7]   7.5: 8.3 | 7.0 | 6.6 | 6.9
//    262144 [13.5] 12.6: 15.7 | 12.7 | 11.8 | 11.3
// (the last row 5 bodies).  Orbits up to e = 0.9, whose groups differ most, want more
// warps: 57344 particles take 10.9 ms plain and 12.2 at 2 warps, 81920 12.9 and 14.1 at 3, 90112
// 19.2 and 15.3 at 3.  So task mode starts at three warps and a tenth more groups than
// warps (64230 live particles).
inline int task_warps_per_partition(int64_t n, int nsteps, int n_sm) {
    const int64_t groups = (n + 31) / 32;
    const int64_t partitions = 4 * (int64_t)std::max(n_sm - 1, 1);
    if (nsteps < 2 * kSubSteps) return 0;
    const int64_t k = std::min<int64_t>(2 + groups / (3 * partitions), kTaskMaxBlocks);
    return k >= 3 && 10 * groups >= 11 * k * partitions ? (int)k : 0;
}

// tb: the task-mode buffers (counter, queue, status), or null for the plain launch.
// force_tasks: task mode whatever the size (two warps per partition at least; GLISSE_LAUNCH_TASKS).
template <int MODE>
cudaError_t launch_particle_chunk_mode(int np, const ChunkArgs& a, const ParticleConsts& pc, cudaStream_t s,
                                       const TaskArgs* tb = nullptr, bool force_tasks = false) {
    if (a.n <= 0) return cudaSuccess;
    SplitConsts sc{};
    split_step_consts(pc, sc);
    for (int j = 0; j < kMaxPlanets; ++j) split_planet(pc, j, sc);
    if constexpr (MODE == kDriftConverge) {
        int dev = 0, nsm = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        int k = tb ? task_warps_per_partition(a.n, a.nsteps, nsm) : 0;
        if (tb && force_tasks && k == 0) k = 2;
        if (k > 0) {
            TaskArgs b = *tb;
            b.sub_steps = task_sub_steps(a.nsteps);
            b.n_groups = (int32_t)((a.n + 31) / 32);
            e = cudaMemsetAsync(b.task_counter, 0, sizeof(unsigned long long), s);
            const size_t n_sub = (size_t)((a.nsteps + b.sub_steps - 1) / b.sub_steps);
            if (e == cudaSuccess)
                e = cudaMemsetAsync(b.queue, 0, sizeof(uint32_t) * (2 + (size_t)b.n_groups * (n_sub - 1)), s);
            if (e != cudaSuccess) return e;
            // k blocks of four warps per SM, one SM's worth short (the ephemeris holds one)
            const int64_t grid = (int64_t)k * std::max(nsm - 1, 1);
            size_t smem = 0;
            switch (np) {
#define GLISSE_TCASE(N)                                                                                  \
    case N:                                                                                              \
        e = particle_smem_cap(reinterpret_cast<const void*>(particle_tasks_kernel<N>), grid, &smem);     \
        if (e != cudaSuccess) return e;                                                                  \
        particle_tasks_kernel<N><<<(unsigned)grid, kParticleBlock, smem, s>>>(a, pc, sc, b);             \
        break;
                GLISSE_TCASE(0)
                GLISSE_TCASE(1)
                GLISSE_TCASE(2)
                GLISSE_TCASE(3)
                GLISSE_TCASE(4)
                GLISSE_TCASE(5)
                GLISSE_TCASE(6)
                GLISSE_TCASE(7)
                GLISSE_TCASE(8)
#undef GLISSE_TCASE
                default: return cudaErrorInvalidValue;
            }
            return cudaGetLastError();
        }
    }
    const int64_t grid = (a.n + kParticleBlock - 1) / kParticleBlock;
    size_t smem = 0;
    cudaError_t e = cudaSuccess;
    switch (np) {
#define GLISSE_CASE(N)                                                                                    \
    case N:                                                                                               \
        e = particle_smem_cap(reinterpret_cast<const void*>(particle_chunk_kernel<N, MODE>), grid, &smem); \
        if (e != cudaSuccess) return e;                                                                   \
        particle_chunk_kernel<N, MODE><<<(unsigned)grid, kParticleBlock, smem, s>>>(a, pc, sc);           \
        break;
        GLISSE_CASE(0)
        GLISSE_CASE(1)
        GLISSE_CASE(2)
        GLISSE_CASE(3)
        GLISSE_CASE(4)
        GLISSE_CASE(5)
        GLISSE_CASE(6)
        GLISSE_CASE(7)
        GLISSE_CASE(8)
#undef GLISSE_CASE
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace glisse
