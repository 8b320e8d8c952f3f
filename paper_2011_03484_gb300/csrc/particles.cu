// particles.cu -- instantiates the test-particle map (particle_map.cuh) with the
// converged fast Kepler solver, and the persistent kernel of batched systems.
#include "particle_map.cuh"

namespace glisse {

// ---------------------------------------------------------------------------
// Batched systems: a persistent kernel.  Each warp takes the next task (a group of 32
// particles of one system over one sub-chunk, handed out as in particle_tasks_kernel),
// stages its system's constants in a warp-private slot of shared memory and runs
// advance_lane with that system's planet count.  One code serves every count: with one
// per count (420 KB) warps of different systems waited a quarter of their time for
// instructions.  When the groups do not outnumber the resident warps, a task is a
// group's whole chunk.
// ---------------------------------------------------------------------------
// TPP = 1: lane k holds particle start + k.  TPP = 2: the lane pair (2k, 2k + 1)
// holds particle start + k (half of the task's 32 particles per call; `half`
// picks which), and only its even lane writes results and counts.
template <int TPP>
__device__ __forceinline__ void batch_task(const BatchArgs& a, const ParticleConsts& pc, const SplitConsts& sc, int s,
                                           int64_t start, int cnt, int lane, int64_t step0, int k0, int m,
                                           bool last, bool test_first, int half) {
    const int np = a.np_of[s];
    const int slot = TPP == 2 ? 16 * half + (lane >> 1) : lane;
    const bool owner = TPP == 1 || (lane & 1) == 0;
    const int64_t i = start + slot;
    const bool in = slot < cnt;
    const int64_t ld = a.ld;
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
    advance_lane<kAnyNp, kDriftConverge, TPP>(pc, sc, a.log + a.log_off[s] + (size_t)k0 * log_stride(np), step0 + k0, m,
                                              test_first && k0 == 0, x, y, z, vx, vy, vz, act, reason, rstep, k0 > 0,
                                              last, PublishTo{}, np);
    if (last) {
        const unsigned live = __reduce_add_sync(kFullMask, (act && owner) ? 1u : 0u);
        if (lane == 0 && live) atomicAdd(reinterpret_cast<unsigned long long*>(a.cnt_new + s), (unsigned long long)live);
    }
    if (a.steps_done) {
        const unsigned adv = (!started || !owner) ? 0u : (rstep >= 0 ? (unsigned)(rstep - (step0 + k0)) : (unsigned)m);
        const unsigned wsum = __reduce_add_sync(kFullMask, adv);
        if (lane == 0 && wsum) atomicAdd(a.steps_done, (unsigned long long)wsum);
    }
    if (in && owner) {
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
}

constexpr int kBatchMaxWarps = 8;  // largest block of the batched kernel: 256 threads

template <int TPP>
__global__ void __launch_bounds__(32 * kBatchMaxWarps, 2) batch_particle_kernel(const BatchArgs a) {
    __shared__ ParticleConsts s_pc[kBatchMaxWarps];
    __shared__ SplitConsts s_sc[kBatchMaxWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n_groups = *a.n_tasks;
    const int64_t step0 = a.clock->step;
    const bool test_first = a.clock->test_first != 0;
    // sub-chunks when the groups outnumber the resident warps by a quarter
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const bool cut = 4 * n_groups >= 5 * warps;
    const int sub = cut ? task_sub_steps(a.nsteps) : a.nsteps;
    const int n_sub = (a.nsteps + sub - 1) / sub;
    constexpr int kWords = (int)(sizeof(ParticleConsts) / sizeof(double));
    static_assert(sizeof(ParticleConsts) % sizeof(double) == 0, "constants must be whole doubles");
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(a.counter, 1);
        t = __shfl_sync(kFullMask, t, 0);
        if (t >= n_groups * n_sub) break;
        int64_t g;
        int k;
        const TaskState got = task_of_ticket(t, n_groups, a.queue, 0, g, k);
        if (got == kTaskTimeout && lane == 0) atomicExch(a.status, GLISSE_E_TIMEOUT);
        if (got != kTaskReady) break;
        const int s = a.task_sys[g];
        const int64_t start = a.task_start[g];
        const int cnt = a.task_count[g];
        const double* src = reinterpret_cast<const double*>(a.pcs + s);
        double* dst = reinterpret_cast<double*>(&s_pc[warp]);
        for (int w = lane; w < kWords; w += 32) dst[w] = src[w];
        __syncwarp();
        if (lane < kMaxPlanets) split_planet(s_pc[warp], lane, s_sc[warp]);
        if (lane == kMaxPlanets) split_step_consts(s_pc[warp], s_sc[warp]);
        __syncwarp();
        do {
#pragma unroll 1
            for (int h = 0; h < TPP; ++h)
                batch_task<TPP>(a, s_pc[warp], s_sc[warp], s, start, cnt, lane, step0, k * sub,
                                min(sub, a.nsteps - k * sub), k + 1 == n_sub, test_first, h);
        } while (task_done(a.queue, a.counter, g, k++, n_sub, n_groups, warps));
    }
}

// Persistent launch: `blocks` blocks of `threads` threads (a multiple of 32, <= 256),
// tpp (1 or 2) lanes per particle.
cudaError_t launch_batch_particles(const BatchArgs& a, int blocks, int threads, int tpp, cudaStream_t s) {
    if (threads < 32 || threads > 32 * kBatchMaxWarps || threads % 32) return cudaErrorInvalidValue;
    if (tpp == 2)
        batch_particle_kernel<2><<<blocks, threads, 0, s>>>(a);
    else if (tpp == 1)
        batch_particle_kernel<1><<<blocks, threads, 0, s>>>(a);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t batch_particles_occupancy(int threads, int tpp, int* blocks_per_sm) {
    if (tpp == 2)
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, batch_particle_kernel<2>, threads, 0);
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, batch_particle_kernel<1>, threads, 0);
}

cudaError_t launch_particle_chunk(int np, const ChunkArgs& a, const ParticleConsts& pc, cudaStream_t s,
                                  const TaskArgs* tb, bool force_tasks) {
    return launch_particle_chunk_mode<kDriftConverge>(np, a, pc, s, tb, force_tasks);
}

// Self-test of the task launch's bounded wait.  Two groups of 32 slots, two sub-chunks;
// the task counter starts past the first sub-chunk of both groups, so each task handed out
// waits for a queue entry that no task appends: its warp gives up after `polls` polls, sets
// *status to GLISSE_E_TIMEOUT and leaves before touching a particle (the other warps find
// no task left).  scratch: zeroed device memory holding the task counter (8 bytes) and
// the queue (16 bytes); the particle arrays point at it too, never read.
cudaError_t particle_wait_selftest(int polls, char* scratch, int* status, cudaStream_t s) {
    constexpr int kGroups = 2;
    ChunkArgs a{};
    a.n = 32 * kGroups;
    a.ld = a.n;
    a.nsteps = 2 * kSubSteps;
    a.log = reinterpret_cast<const double*>(scratch);
    a.st = reinterpret_cast<double*>(scratch);
    a.id = reinterpret_cast<const int32_t*>(scratch);
    a.alive = reinterpret_cast<uint8_t*>(scratch);
    TaskArgs ta{};
    ta.sub_steps = kSubSteps;
    ta.n_groups = kGroups;
    ta.task_counter = reinterpret_cast<unsigned long long*>(scratch);
    ta.queue = reinterpret_cast<uint32_t*>(scratch + 8);
    ta.status = status;
    ta.wait_polls = polls;
    const unsigned long long first = kGroups;
    cudaError_t e = cudaMemcpyAsync(ta.task_counter, &first, sizeof(first), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    particle_tasks_kernel<0><<<4, kParticleBlock, 0, s>>>(a, ParticleConsts{}, SplitConsts{}, ta);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e;
}

}  // namespace glisse
