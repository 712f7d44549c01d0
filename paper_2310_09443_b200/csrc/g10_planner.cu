// Algorithm 1 (smart tensor eviction) as printed: one persistent cooperative kernel in which every
// iteration rescores all live inactive periods in parallel, reduces the best benefit/cost ratio across the
// grid, commits it and tests the peak -- two grid barriers per iteration, no host round trip.  Selected by
// G10_FLAG_RESCORE_ALL; the other planners give the same plan with far less work: one cluster (g10_planner_chip.cu), all SMs'
// shared memory (g10_planner_spread.cu) or global memory (g10_planner_lazy.cu), whichever the trace fits first.
#include "g10_planner.cuh"

namespace g10 {

// kCyclic: steady-state planning (period and geometry arrays hold slots unrolled over two iterations, A.start is the
// unrolled clock; see phys_slot) for traces too large for the on-chip planner, which runs first: when it has
// produced the plan (`done`), this grid returns at once.
template <bool kCyclic>
__global__ void __launch_bounds__(kPlanThreads, 1) k_plan_loop(PlanArgs A, const unsigned *done)
{
    if (kCyclic && *done) return;          // (same answer in every thread of the grid: written by an earlier launch)
    if (kCyclic && blockIdx.x == 0 && threadIdx.x == 0) A.summary[7] = 0;      // (the on-chip planner may have left "does not fit" there)
    __shared__ Cand s_cand[kPlanWarps + 1];
    __shared__ long long s_max[kPlanWarps + 1];
    const int G = gridDim.x, c = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t Pn = *A.Pn_dev < A.geo_stride ? *A.Pn_dev : A.geo_stride;
    const int64_t limit = (A.max_iterations <= 0 || A.max_iterations > Pn) ? Pn : A.max_iterations;
    unsigned gen = 0;
    int64_t n_mig = 0, rounds = 0, bytes_ssd = 0, bytes_host = 0;
    int status = -1;
    bool own_dirty = true;
    long long peak = 0;

    for (int64_t it = 0;; ++it) {
        if (own_dirty) {
            const long long m = own_slots_max(A, c, G, s_max);
            if (threadIdx.x == 0) A.peak_part[c] = m;
            own_dirty = false;
        }
        // ---- score: one warp per live period
        Cand best;
        best.ben = 0; best.cost = 1; best.idx = -1; best.dest = -1;
        for (int64_t p = (int64_t)c * kPlanWarps + warp; p < Pn; p += (int64_t)G * kPlanWarps) {
            if (A.dead[p]) continue;
            Cand cd;
            if (!score_period<kCyclic>(A, p, lane, &cd)) {
                if (lane == 0) A.dead[p] = 1;       // channels only fill up: never admissible again
                continue;
            }
            if (lane == 0 && cd.ben > 0 && cand_beats(cd, best)) best = cd;
        }
        best = block_best(best, s_cand);
        if (threadIdx.x == 0) {
            Proposal pr;
            pr.ben_lo = (ull)best.ben; pr.ben_hi = (ull)(best.ben >> 64); pr.cost = best.cost; pr.idx = best.idx; pr.dest = best.dest;
            A.proposals[c] = pr;
        }
        if (!grid_barrier(A.bar, G, gen)) { status = -2; break; }

        // ---- reduce peak and proposals (every block, redundantly and identically)
        long long m = 0;
        Cand w;
        w.ben = 0; w.cost = 1; w.idx = -1; w.dest = -1;
        for (int j = threadIdx.x; j < G; j += kPlanThreads) {
            const long long pm = __ldcg(&A.peak_part[j]);
            if (pm > m) m = pm;
            Cand x;
            const ull lo = __ldcg(&A.proposals[j].ben_lo), hi = __ldcg(&A.proposals[j].ben_hi);
            x.ben = ((u128)hi << 64) | lo;
            x.cost = __ldcg(&A.proposals[j].cost);
            x.idx = __ldcg(&A.proposals[j].idx);
            x.dest = __ldcg(&A.proposals[j].dest);
            if (cand_beats(x, w)) w = x;
        }
        peak = block_max_i64(m, s_max);
        const Cand win = block_best(w, s_cand);
        if (A.fits_always || peak <= A.cap) { status = n_mig == 0 ? G10_ALREADY_FITS : G10_FIT; break; }
        if (it >= limit) { status = limit < Pn ? G10_ITERATION_LIMIT : G10_EXHAUSTED; break; }
        rounds += 1;
        if (win.idx < 0) { status = G10_EXHAUSTED; break; }

        int64_t sz = 0;
        if (commit_winner<kCyclic>(A, win.idx, win.dest, it, n_mig, c, G, &sz)) own_dirty = true;
        n_mig += 1;
        if (win.dest == G10_DEST_SSD) bytes_ssd += sz; else bytes_host += sz;
        if (!grid_barrier(A.bar, G, gen)) { status = -2; break; }
    }
    plan_epilogue(A, c, G, gen, status, peak, n_mig, rounds, bytes_ssd, bytes_host);
}

// copies the device status word into summary[7] / counts[2] / *status once everything before it ran
__global__ void k_publish_status(const ull *status, int64_t *dst) { *dst = (int64_t)*status; }

cudaError_t launch_publish_status(const Workspace &w, int64_t *dst, cudaStream_t s)
{
    k_publish_status<<<1, 1, 0, s>>>(w.status, dst); count_launch();
    return cudaGetLastError();
}

void fill_plan_args(const DeviceTrace &t, const Workspace &w, const PlanParams &p, PlanArgs &A)
{
    A.K = t.K;
    A.Pn_dev = w.counts + 1;
    A.geo_stride = t.E > 0 ? t.E : 1;
    A.start = w.start; A.dur = t.kernel_ns; A.bytes = t.tensor_bytes;
    A.per_t = w.period_tensor; A.per_u = w.period_prev_use; A.per_v = w.period_next_use;
    A.geo_t = w.geo_t; A.geo_a = w.geo_a; A.geo_b = w.geo_b;
    A.P = p.final_pressure; A.busy = w.busy; A.hocc = w.hocc; A.dead = w.dead;
    A.fits_always = p.gpu_capacity_bytes >= ((uint64_t)1 << 63) ? 1 : 0;
    A.cap = A.fits_always ? INT64_MAX : (int64_t)p.gpu_capacity_bytes;
    A.bw[G10_DEST_SSD] = p.ssd_bw; A.bw[G10_DEST_HOST] = p.host_bw;
    A.host_capacity = p.host_capacity_bytes;
    A.max_iterations = p.max_iterations;
    A.out = p.migrations; A.out_cap = p.migrations_cap; A.summary = p.summary;
    A.proposals = w.proposals; A.peak_part = w.peak_part; A.peak_key = w.peak_key;
    A.bar = (GridBarrier *)w.barrier; A.status = w.status;
}

static int blocks_for(const void *kernel)
{
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kPlanThreads, 0) != cudaSuccess) return 0;
    if (per_sm < 1) return 0;
    return sms > kMaxPlanBlocks ? kMaxPlanBlocks : sms;      // one block per SM
}

cudaError_t launch_plan_lazy(const PlanArgs &A, const Workspace &w, int G, cudaStream_t s);
int plan_lazy_blocks();
bool plan_spread_possible(int64_t K, int64_t E);
cudaError_t launch_plan_spread(const PlanArgs &A, const Workspace &w, cudaStream_t s);
int plan_chip_blocks(int64_t E, bool several, bool cyclic);
int plan_chip_possible(int64_t K, int64_t E, int C, bool host_cap, bool cyclic);
cudaError_t launch_plan_chip(const PlanArgs &A, const Workspace &w, int C, bool cyclic, bool alone, cudaStream_t s);

static int chip_blocks(int64_t E, uint32_t flags, bool cyclic) { return plan_chip_blocks(E, (flags & G10_FLAG_MULTI_BLOCK) != 0, cyclic); }

bool plan_keeps_state_on_chip(int64_t K, int64_t E, bool host_cap, uint32_t flags, bool cyclic)
{
    if (flags & (G10_FLAG_RESCORE_ALL | G10_FLAG_GLOBAL_STATE | G10_FLAG_SPREAD_STATE)) return false;
    return plan_chip_possible(K, E, chip_blocks(E, flags, cyclic), host_cap, cyclic) == 2;
}

cudaError_t launch_plan_batch(const PlanArgs &A, const Workspace &w, int V, int C, const BatchArgs &B, int64_t *stability, cudaStream_t s);

cudaError_t launch_plan_variants(const DeviceTrace &t, const Workspace &w, const PlanParams &p, int V, int C, int64_t *stability, cudaStream_t s)
{
    PlanArgs A;
    fill_plan_args(t, w, p, A);
    BatchArgs B;
    B.variants = w.batch_variants; B.P0 = w.pressure; B.P_out = p.final_pressure; B.host_cap = p.host_capacity_bytes != 0 ? 1 : 0;
    return launch_plan_batch(A, w, V, C, B, stability, s);
}

cudaError_t launch_plan_cyclic(const DeviceTrace &t, const Workspace &w, const PlanParams &p, cudaStream_t s)
{
    PlanArgs A;
    fill_plan_args(t, w, p, A);
    A.start = w.start2;
    // one cluster plans when everything fits its shared memory; where only the device can tell, the planner that uses the whole
    // GPU is queued behind it and does the work otherwise
    const int C = chip_blocks(t.E, 0, true), fits = plan_chip_possible(t.K, t.E, C, p.host_capacity_bytes != 0, true);
    if (fits) {
        const cudaError_t e = launch_plan_chip(A, w, C, true, fits == 2, s);
        if (e != cudaSuccess || fits == 2) return e;
    }
    const int G = blocks_for((const void *)k_plan_loop<true>);
    if (G < 1) return cudaErrorLaunchFailure;
    const unsigned *done = w.one_done;
    void *args[] = {&A, &done};
    return cudaLaunchCooperativeKernel((const void *)k_plan_loop<true>, dim3(G), dim3(kPlanThreads), args, 0, s);
}

// ORs the call's status word into *dst (which the planner may already have written)
__global__ void k_publish_status_or(const ull *status, int64_t *dst) { *dst |= (int64_t)*status; }

cudaError_t launch_publish_status_or(const Workspace &w, int64_t *dst, cudaStream_t s)
{
    k_publish_status_or<<<1, 1, 0, s>>>(w.status, dst); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_plan_loop(const DeviceTrace &t, const Workspace &w, const PlanParams &p, cudaStream_t s)
{
    PlanArgs A;
    fill_plan_args(t, w, p, A);
    if (p.flags & G10_FLAG_RESCORE_ALL) {
        const int G = blocks_for((const void *)k_plan_loop<false>);
        if (G < 1) return cudaErrorLaunchFailure;
        const unsigned *done = w.one_done;
        void *args[] = {&A, &done};
        return cudaLaunchCooperativeKernel((const void *)k_plan_loop<false>, dim3(G), dim3(kPlanThreads), args, 0, s);
    }
    if (!(p.flags & (G10_FLAG_GLOBAL_STATE | G10_FLAG_SPREAD_STATE))) {
        // (as in launch_plan_cyclic)
        const int C = chip_blocks(t.E, p.flags, false), fits = plan_chip_possible(t.K, t.E, C, p.host_capacity_bytes != 0, false);
        if (fits) {
            const cudaError_t e = launch_plan_chip(A, w, C, false, fits == 2, s);
            if (e != cudaSuccess || fits == 2) return e;
        }
    }
    // state spread over the shared memory of all SMs if it fits (the device knows), else in global memory
    if (!(p.flags & G10_FLAG_GLOBAL_STATE) && plan_spread_possible(t.K, t.E)) {
        const cudaError_t e = launch_plan_spread(A, w, s);
        if (e != cudaSuccess) return e;
    }
    const int G = plan_lazy_blocks();
    if (G < 1) return cudaErrorLaunchFailure;
    return launch_plan_lazy(A, w, G, s);
}

}  // namespace g10
