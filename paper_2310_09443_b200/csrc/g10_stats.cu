// Workload characterisation (Section 3, Figures 2-4) from the vitality results of a trace:
//   active_bytes[k]  bytes of the tensors kernel k uses (the working set of Figure 2),
//   len_hist         inactive periods by floor(log2(length in ns))            (Figure 3),
//   size_len_hist    periods by floor(log2 size) x floor(log2 length)         (Figure 4),
//   hide             periods long enough for a round trip to the SSD / the host memory, 2 t <= L.
// The per-kernel sums go through the per-tensor use lists (already free of duplicates), one 64-bit atomic per
// (kernel, tensor) incidence; the histograms are counted in shared memory and flushed once per block.
// Three launches, each placed while its predecessor drains: clear the outputs; per-kernel sums and histograms side by side in one
// grid (both are bound by the L2's rate of scattered 32-byte requests, 1.4 M reductions and 0.8 M loads on 1.1 M tensors); maximum
// and arg-max by one cluster of 16 blocks, which needs no scratch.  Four kernels and five memsets took 38 us where this takes 21.
#include "g10_device.cuh"
#include "g10_internal.h"

namespace g10 {

constexpr int kStatThreads = 256;
constexpr int kLenBins = 64, kSizeBins = 41, kLen2Bins = 45;

constexpr int kPeakThreads = 1024;
constexpr long long kNone = 0x7fffffffffffffffll;

struct StatsOut {
    ull *active, *len_hist, *size_len_hist, *hide;
    long long *summary;
};

__global__ void __launch_bounds__(kStatThreads) k_stats_clear(int64_t K, StatsOut out)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t me = (int64_t)blockIdx.x * kStatThreads + threadIdx.x, all = (int64_t)gridDim.x * kStatThreads;
    for (int64_t k = me; k < K; k += all) out.active[k] = 0;
    for (int64_t b = me; b < kSizeBins * kLen2Bins; b += all) out.size_len_hist[b] = 0;
    if (me < kLenBins) out.len_hist[me] = 0;
    if (me < 2) out.hide[me] = 0;
}

__device__ __forceinline__ int floor_log2(long long x) { return x > 1 ? 63 - __clzll(x) : 0; }

// Blocks [0, period_blocks): histograms of the periods; the others: bytes per kernel.
__global__ void __launch_bounds__(kStatThreads) k_stats(int64_t N, const int64_t *__restrict__ use_ptr, const int32_t *__restrict__ uses,
                                                        const int64_t *__restrict__ bytes, const int64_t *__restrict__ start, int64_t Pn,
                                                        const int32_t *__restrict__ per_t, const int32_t *__restrict__ per_u,
                                                        const int32_t *__restrict__ per_v, uint64_t host_bw, uint64_t ssd_bw, int period_blocks,
                                                        StatsOut out)
{
    __shared__ unsigned s_len[kLenBins];
    __shared__ unsigned s_sl[kSizeBins * kLen2Bins];
    __shared__ unsigned s_hide[2];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31;
    if ((int)blockIdx.x >= period_blocks) {
        const int64_t nthreads = (int64_t)(gridDim.x - period_blocks) * kStatThreads;
        const int64_t first = (int64_t)(blockIdx.x - period_blocks) * kStatThreads + (threadIdx.x & ~31);
        bool waited = false;
        for (int64_t base = first; base < N; base += nthreads) {
            const int64_t i = base + lane;
            int64_t lo = 0, hi = 0;
            ull s = 0;
            if (i < N) { lo = use_ptr[i]; hi = use_ptr[i + 1]; s = (ull)bytes[i]; }
            if (!waited) { asm volatile("griddepcontrol.wait;" ::: "memory"); waited = true; }      // (the outputs are cleared)
            const bool heavy = hi - lo > 64;
            if (!heavy) for (int64_t j = lo; j < hi; ++j) atomicAdd(&out.active[uses[j]], s);
            unsigned m = __ballot_sync(0xffffffffu, heavy);
            while (m) {                                   // a tensor with a long use list: the warp shares it
                const int src = __ffs(m) - 1;
                m &= m - 1;
                const int64_t l2 = __shfl_sync(0xffffffffu, lo, src), h2 = __shfl_sync(0xffffffffu, hi, src);
                const ull s2 = __shfl_sync(0xffffffffu, s, src);
                for (int64_t j = l2 + lane; j < h2; j += 32) atomicAdd(&out.active[uses[j]], s2);
            }
        }
        if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    for (int b = threadIdx.x; b < kLenBins; b += kStatThreads) s_len[b] = 0;
    for (int b = threadIdx.x; b < kSizeBins * kLen2Bins; b += kStatThreads) s_sl[b] = 0;
    if (threadIdx.x < 2) s_hide[threadIdx.x] = 0;
    __syncthreads();
    unsigned h0 = 0, h1 = 0;
    constexpr int kAhead = 2;                            // periods of a thread whose loads are in flight together
    const int64_t step = (int64_t)period_blocks * kStatThreads;
    for (int64_t p0 = (int64_t)blockIdx.x * kStatThreads + threadIdx.x; p0 < Pn; p0 += kAhead * step) {
        int32_t t[kAhead], u[kAhead], v[kAhead];
        long long L[kAhead], s[kAhead];
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            const int64_t p = p0 + q * step;
            t[q] = p < Pn ? per_t[p] : -1; u[q] = p < Pn ? per_u[p] : 0; v[q] = p < Pn ? per_v[p] : 0;
        }
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            L[q] = 0; s[q] = 0;
            if (t[q] >= 0) { L[q] = start[v[q]] - start[u[q] + 1]; s[q] = bytes[t[q]]; }
        }
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            if (t[q] < 0) continue;
            const int bl = floor_log2(L[q]), bs = floor_log2(s[q]);
            atomicAdd(&s_len[bl], 1u);
            atomicAdd(&s_sl[min(bs, kSizeBins - 1) * kLen2Bins + min(bl, kLen2Bins - 1)], 1u);
            // ceil(s * 1e9 / bw) <= L / 2  <=>  s * 1e9 <= (L / 2) * bw
            const u128 need = (u128)(ull)s[q] * (u128)1000000000ull, half = (u128)(ull)(L[q] / 2);
            h0 += need <= half * (u128)ssd_bw;
            h1 += need <= half * (u128)host_bw;
        }
    }
    h0 = __reduce_add_sync(0xffffffffu, h0);
    h1 = __reduce_add_sync(0xffffffffu, h1);
    if (lane == 0) { if (h0) atomicAdd(&s_hide[0], h0); if (h1) atomicAdd(&s_hide[1], h1); }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int b = threadIdx.x; b < kLenBins; b += kStatThreads) if (s_len[b]) atomicAdd(&out.len_hist[b], (ull)s_len[b]);
    for (int b = threadIdx.x; b < kSizeBins * kLen2Bins; b += kStatThreads) if (s_sl[b]) atomicAdd(&out.size_len_hist[b], (ull)s_sl[b]);
    if (threadIdx.x < 2 && s_hide[threadIdx.x]) atomicAdd(&out.hide[threadIdx.x], (ull)s_hide[threadIdx.x]);
}

// summary = largest active bytes, its lowest kernel (0, -1 for an empty trace).  One cluster, the largest that the
// device can place; every block reads every kBlocks-th run.  (One kernel with its size given at launch: a microsecond more.)
template <int kBlocks>
__global__ void __launch_bounds__(kPeakThreads) __cluster_dims__(kBlocks, 1, 1) k_active_peak(int64_t K, const long long *__restrict__ active, long long *summary)
{
    __shared__ long long s_mx[kPeakThreads / 32], s_at[kPeakThreads / 32];
    __shared__ longlong2 s_all[kBlocks];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int64_t step = (int64_t)kBlocks * kPeakThreads;
    auto better = [](long long m, long long a, long long &mx, long long &at) { if (m > mx || (m == mx && a < at)) { mx = m; at = a; } };
    long long mx = -1, at = kNone;
    // (a block's shared memory may be written by others once it has started, not before: all say that they have, and wait for it
    // where the first remote store stands)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t k0 = (int64_t)blockIdx.x * kPeakThreads + threadIdx.x; k0 < K; k0 += 8 * step) {
        long long v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) { const int64_t k = k0 + q * step; v[q] = k < K ? __ldcg(&active[k]) : -1; }
#pragma unroll
        for (int q = 0; q < 8; ++q) if (v[q] > mx) { mx = v[q]; at = k0 + q * step; }    // (k ascending: the first stays)
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long ym = __shfl_xor_sync(0xffffffffu, mx, o), ya = __shfl_xor_sync(0xffffffffu, at, o);
        better(ym, ya, mx, at);
    }
    if (lane == 0) { s_mx[warp] = mx; s_at[warp] = at; }
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 0) {
        mx = s_mx[lane]; at = s_at[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long ym = __shfl_xor_sync(0xffffffffu, mx, o), ya = __shfl_xor_sync(0xffffffffu, at, o);
            better(ym, ya, mx, at);
        }
        if (lane == 0) {                                  // into the first block's shared memory
            unsigned dst;
            asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"((unsigned)__cvta_generic_to_shared(&s_all[blockIdx.x])));
            asm volatile("st.shared::cluster.v2.b64 [%0], {%1, %2};" ::"r"(dst), "l"(mx), "l"(at) : "memory");
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int b = 1; b < kBlocks; ++b) better(s_all[b].x, s_all[b].y, mx, at);
        summary[0] = K > 0 ? mx : 0; summary[1] = K > 0 ? at : -1;
    }
}

static int stat_grid(int64_t items, int per_block)
{
    int64_t g = (items + per_block - 1) / per_block;
    const int64_t cap = 148 * 8;
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

cudaError_t launch_characterize(int64_t K, int64_t N, const int64_t *use_ptr, const int32_t *uses, const int64_t *bytes, const int64_t *start,
                                int64_t Pn, const int32_t *per_t, const int32_t *per_u, const int32_t *per_v, uint64_t host_bw, uint64_t ssd_bw,
                                int64_t *active, int64_t *len_hist, int64_t *size_len_hist, int64_t *hide, int64_t *summary, cudaStream_t s)
{
    static int known[kMaxDevices];
    cudaError_t e;
    StatsOut out{(ull *)active, (ull *)len_hist, (ull *)size_len_hist, (ull *)hide, (long long *)summary};
    k_stats_clear<<<stat_grid(K > 2 * kSizeBins * kLen2Bins ? K : 2 * kSizeBins * kLen2Bins, 2 * kStatThreads), kStatThreads, 0, s>>>(K, out); count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s; cfg.attrs = at; cfg.numAttrs = 1; cfg.blockDim = dim3(kStatThreads);
    const int pb = Pn > 0 ? stat_grid(Pn, kStatThreads * 2) : 0, tb = N > 0 && K > 0 ? stat_grid(N, kStatThreads) : 0;
    if (pb + tb > 0) {
        cfg.gridDim = dim3((unsigned)(pb + tb));
        if ((e = cudaLaunchKernelEx(&cfg, k_stats, N, use_ptr, uses, bytes, start, Pn, per_t, per_u, per_v, host_bw, ssd_bw, pb, out)) != cudaSuccess) return e;
    }
    void (*const peak[])(int64_t, const long long *, long long *) = {k_active_peak<16>, k_active_peak<8>, k_active_peak<4>, k_active_peak<2>, k_active_peak<1>};
    const void *const any[] = {(const void *)peak[0], (const void *)peak[1], (const void *)peak[2], (const void *)peak[3], (const void *)peak[4]};
    const int most = largest_cluster(any, true, kPeakThreads, 0, known);
    int j = 0;
    while (j < 4 && 16 >> j > most) ++j;
    cfg.gridDim = dim3(16u >> j); cfg.blockDim = dim3(kPeakThreads);
    if ((e = allow_launch(any[j], 0, 16 >> j)) != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, peak[j], K, (const long long *)active, (long long *)summary);
}

}  // namespace g10
