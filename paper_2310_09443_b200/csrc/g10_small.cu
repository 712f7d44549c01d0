// All of the analysis -- slot clock, tensor vitality, pressure timeline, and for the steady-state planner the unrolled clock and
// the wrap-around periods -- of a trace that fits the shared memory of one SM, by ONE block in one launch.  The general passes are
// five launches of a few microseconds each on such a trace, every one a chain of latencies on a nearly idle GPU; here a step hands
// over to the next through shared memory and a block barrier.  Inputs are read once and outputs written once, both coalesced, so
// that the pointers may also be those of pinned host memory: no copies, no staging.
// Kernels, tensors and positions in the use lists are 16-bit numbers in shared memory (K, N, E < 65535).
#include "g10_device.cuh"
#include "g10_internal.h"

namespace g10 {

constexpr int kSmThreads = 1024;
constexpr int kSmWarps = kSmThreads / 32;
constexpr int kSmMid = 32;                          // longer segments are sorted by a warp or by the block
constexpr int kSmWarpSort = 1024;                   // ... up to this length by a warp
typedef unsigned short u16;

struct SmallLayout {
    size_t r1, r2, r3, off, dp, total;              // byte offsets of the regions
};
__host__ __device__ inline SmallLayout small_layout(int64_t K, int64_t N, int64_t E)
{
    auto up = [](size_t x) { return (x + 15) / 16 * 16; };
    const size_t ev = up((size_t)E * 2), slots = up((size_t)(K + 1) * 8), a = ev > slots ? ev : slots;
    SmallLayout l;
    l.r1 = 0; l.r2 = a; l.r3 = 2 * a; l.off = l.r3 + ev; l.dp = l.off + up((size_t)(N + 1) * 4); l.total = l.dp + up((size_t)(N + 1) * 4);
    return l;
}

// Exclusive sum over the block (one value per thread); *total gets the sum of all.
template <typename T>
__device__ __forceinline__ T small_scan(T v, T *s_w /* [kSmWarps] */, T *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const T y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
    __syncthreads();                                // (s_w free)
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    const T x = s_w[lane];
    T xi = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const T y = __shfl_up_sync(0xffffffffu, xi, o); if (lane >= o) xi += y; }
    *total = __shfl_sync(0xffffffffu, xi, 31);
    return __shfl_sync(0xffffffffu, xi - x, warp) + incl - v;
}

// In-place exclusive prefix of n entries in shared memory: a run of consecutive entries per thread (an odd number, so that the
// threads of a warp meet in different banks).  Returns the total; ends without a barrier.
template <typename T>
__device__ __forceinline__ T small_prefix(T *a, int n, T *s_w)
{
    const int c = ((n + kSmThreads - 1) / kSmThreads) | 1, lo = (int)threadIdx.x * c < n ? (int)threadIdx.x * c : n, hi = lo + c < n ? lo + c : n;
    T sum = 0, total;
#pragma unroll 4
    for (int k = lo; k < hi; ++k) sum += a[k];
    T run = small_scan<T>(sum, s_w, &total);
#pragma unroll 4
    for (int k = lo; k < hi; ++k) { const T v = a[k]; a[k] = run; run += v; }
    return total;
}

// Adds to a 64-bit word of shared memory: two 32-bit atomics with a carry (a 64-bit one is a compare-and-swap loop).
__device__ __forceinline__ void small_add64(long long *p, long long v)
{
    unsigned *w = reinterpret_cast<unsigned *>(p);
    const unsigned lo = (unsigned)v, old = atomicAdd(&w[0], lo);
    const unsigned up = (unsigned)((ull)v >> 32) + (old + lo < old ? 1u : 0u);
    if (up) atomicAdd(&w[1], up);
}

// Largest value of the lanes and its lowest slot (slot < 0: the lane has none), in every lane.
__device__ __forceinline__ void small_peak(long long &mx, int &sl)
{
    const unsigned hi = sl >= 0 ? (unsigned)((ull)mx >> 32) ^ 0x80000000u : 0u, lo = sl >= 0 ? (unsigned)mx : 0u;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi), ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const unsigned s = __reduce_min_sync(0xffffffffu, sl >= 0 && hi == mh && lo == ml ? (unsigned)sl : 0xffffffffu);
    mx = (long long)((ull)(mh ^ 0x80000000u) << 32 | ml); sl = (int)s;              // (all ones: -1)
}

// Removes the repeats of a sorted segment and counts its periods (one warp); distinct uses | periods << 16.
__device__ unsigned small_compact_warp(u16 *seg, int m, int lane)
{
    int d = 0, pp = 0, prev = -1;                   // prev: last use kept so far
    for (int c0 = 0; c0 < m; c0 += 32) {
        const int t = c0 + lane;
        const int x = t < m ? seg[t] : 0x10000;
        int before = __shfl_up_sync(0xffffffffu, x, 1);
        if (lane == 0) before = prev;
        const bool keep = t < m && x != before, per = keep && before >= 0 && x - before >= 2;
        const unsigned mk = __ballot_sync(0xffffffffu, keep), mp = __ballot_sync(0xffffffffu, per);
        if (keep) seg[d + __popc(mk & ((1u << lane) - 1u))] = (u16)x;        // (never overtakes an unread entry)
        d += __popc(mk); pp += __popc(mp);
        const int last = (m - c0 < 32 ? m - c0 : 32) - 1;
        prev = __shfl_sync(0xffffffffu, x, last);
        __syncwarp();
    }
    return (unsigned)d | (unsigned)pp << 16;
}

__global__ void __launch_bounds__(kSmThreads, 1) k_small(SmallArgs A)
{
    extern __shared__ __align__(16) unsigned char s_mem[];
    __shared__ long long s_w64[kSmWarps];
    __shared__ unsigned s_w32[kSmWarps];
    __shared__ int s_sl[kSmWarps];
    __shared__ unsigned s_bits;
    __shared__ int s_nmid, s_nheavy;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = (int)A.t.K, N = (int)A.t.N, E = (int)A.t.E;
    const SmallLayout l = small_layout(K, N, E);
    u16 *s_id = (u16 *)(s_mem + l.r1), *s_krel = (u16 *)(s_mem + l.r2), *ks = (u16 *)(s_mem + l.r3);
    long long *s_diff = (long long *)(s_mem + l.r1), *s_ns = (long long *)(s_mem + l.r2);
    unsigned *off = (unsigned *)(s_mem + l.off), *dp = (unsigned *)(s_mem + l.dp);
    const bool clock = A.start != nullptr;
    unsigned bad = 0;

    // ---- tensor ids, durations, kernels of the events.  The first batch of all three arrays (all of them, up to 4096 kernels and
    // 16 384 events) is on its way before anything is used: one round trip instead of three -- a microsecond each from a cold L2,
    // 1.5 from host memory.  (All loads of a batch before the first use: the stores in between would keep the compiler from it.)
    constexpr int kIn = 4;
    const int E4 = ((uintptr_t)A.t.kernel_tensors & 15) == 0 ? E / 4 : 0;        // events taken four at a time
    long long dur[kIn];
    int4 ids[kIn];
    int64_t first[kIn], next[kIn];
    auto load_dur = [&](int k0) {
#pragma unroll
        for (int q = 0; q < kIn; ++q) dur[q] = k0 + q * kSmThreads < K ? A.t.kernel_ns[k0 + q * kSmThreads] : 1;
    };
    auto load_ids = [&](int e0) {
#pragma unroll
        for (int q = 0; q < kIn; ++q) ids[q] = e0 + q * kSmThreads < E4 ? reinterpret_cast<const int4 *>(A.t.kernel_tensors)[e0 + q * kSmThreads] : make_int4(0, 0, 0, 0);
    };
    auto load_ptr = [&](int k0) {                   // (k0: of the warp's first lane)
#pragma unroll
        for (int q = 0; q < kIn; ++q) {
            const int k = k0 + q * kSmThreads + lane;
            first[q] = k <= K ? A.t.kernel_ptr[k] : E;
            next[q] = lane == 31 && k < K ? A.t.kernel_ptr[k + 1] : E;
        }
    };
    if (clock) load_dur(tid);
    load_ids(tid);
    load_ptr(warp * 32);
    if (tid == 0) { s_bits = 0; s_nmid = 0; s_nheavy = 0; }
#pragma unroll 4
    for (int t = tid; t <= N; t += kSmThreads) off[t] = 0;
    __syncthreads();
    if (clock)
        for (int k0 = tid; k0 < K; k0 += kIn * kSmThreads) {
            if (k0 != tid) load_dur(k0);
#pragma unroll
            for (int q = 0; q < kIn; ++q) {
                if (dur[q] < 1 || dur[q] >= ((long long)1 << 44)) { bad |= G10_DEV_BAD_DURATION; dur[q] = 1; }
                if (k0 + q * kSmThreads < K) s_ns[k0 + q * kSmThreads] = dur[q];
            }
        }
    auto event = [&](int e, int id) {
        const bool ok = id >= 0 && id < N;
        if (ok) atomicAdd(&off[id], 1u); else bad |= G10_DEV_BAD_TENSOR_ID;
        s_id[e] = ok ? (u16)id : (u16)0xffff;
    };
    for (int e0 = tid; e0 < E4; e0 += kIn * kSmThreads) {
        if (e0 != tid) load_ids(e0);
#pragma unroll
        for (int q = 0; q < kIn; ++q) {
            const int e = 4 * (e0 + q * kSmThreads);
            if (e < 4 * E4) { event(e, ids[q].x); event(e + 1, ids[q].y); event(e + 2, ids[q].z); event(e + 3, ids[q].w); }
        }
    }
    for (int e = 4 * E4 + tid; e < E; e += kSmThreads) event(e, A.t.kernel_tensors[e]);
    if (clock) {
        // slot clock
        __syncthreads();
        const long long total = small_prefix<long long>(s_ns, K, s_w64);
        if (total >= ((long long)1 << 44)) bad |= G10_DEV_BAD_DURATION;
        __syncthreads();
        for (int k = tid; k < K; k += kSmThreads) {
            const long long s = s_ns[k];
            A.start[k] = s;
            if (A.start2 != nullptr) { A.start2[k] = s; A.start2[K + k] = s + total; }
        }
        if (tid == 0) { A.start[K] = total; if (A.start2 != nullptr) A.start2[2 * K] = 2 * total; }
        __syncthreads();
    }
    // (a kernel_ptr that is no monotone map onto [0, E] leaves every tensor unused; the walk stays inside the events in any case)
    for (int k0 = warp * 32; k0 < K; k0 += kIn * kSmThreads) {
        if (k0 != warp * 32) load_ptr(k0);
#pragma unroll
        for (int q = 0; q < kIn; ++q) {
            const int kq = k0 + q * kSmThreads, k = kq + lane;
            if (kq >= K) break;
            const int64_t p0 = first[q], down = __shfl_down_sync(0xffffffffu, first[q], 1), p1 = lane == 31 ? next[q] : down;
            if (k < K && (p0 > p1 || p0 < 0 || p1 > E || (k == 0 && p0 != 0) || (k == K - 1 && p1 != E))) bad |= G10_DEV_BAD_KERNEL_PTR;
            const int a = p0 < 0 ? 0 : p0 > E ? E : (int)p0, b = k >= K || p1 < 0 ? 0 : p1 > E ? E : (int)p1;
            const bool wide = b - a > 64;
            if (!wide) for (int p = a; p < b; ++p) s_krel[p] = (u16)k;
            unsigned m = __ballot_sync(0xffffffffu, wide);
            while (m) {
                const int src = __ffs(m) - 1;
                m &= m - 1;
                const int wa = __shfl_sync(0xffffffffu, a, src), wb = __shfl_sync(0xffffffffu, b, src);
                for (int p = wa + lane; p < wb; p += 32) s_krel[p] = (u16)(kq + src);
            }
        }
    }
    {
        const unsigned w = __reduce_or_sync(0xffffffffu, bad);
        if (lane == 0 && w) atomicOr(&s_bits, w);
    }
    // ---- events into per-tensor segments of ks (off[t]: first the start of t's segment, after the scatter its end)
    __syncthreads();
    small_prefix<unsigned>(off, N, s_w32);
    __syncthreads();
    const bool none = (s_bits & G10_DEV_BAD_KERNEL_PTR) != 0;
    if (!none)
#pragma unroll 4
        for (int e = tid; e < E; e += kSmThreads) {
            const unsigned id = s_id[e];
            if (id != 0xffffu) ks[atomicAdd(&off[id], 1u)] = s_krel[e];
        }
    __syncthreads();
    u16 *s_mid = s_krel;                            // tensors with three to kSmMid raw uses; with more, from the other end
    auto segment = [&](int t, int *m) {
        const int o = t > 0 ? (int)off[t - 1] : 0;
        *m = none ? 0 : (int)off[t] - o;
        return ks + o;
    };
#pragma unroll 2
    for (int t = tid; t < N; t += kSmThreads) {
        int m;
        u16 *seg = segment(t, &m);
        unsigned r = m > 0 ? 1u : 0u;
        if (m == 2) {
            const int x = seg[0], y = seg[1], lo = x < y ? x : y, hi = x < y ? y : x;
            if (lo != hi) { seg[0] = (u16)lo; seg[1] = (u16)hi; r = 2u | (hi - lo >= 2 ? 1u << 16 : 0u); }
        } else if (m > kSmMid) s_mid[E - 1 - atomicAdd(&s_nheavy, 1)] = (u16)t;
        else if (m > 2) s_mid[atomicAdd(&s_nmid, 1)] = (u16)t;
        dp[t] = r;
    }
    __syncthreads();
    const int nmid = s_nmid, nheavy = s_nheavy;
    for (int q = tid; q < nmid; q += kSmThreads) {
        const int t = s_mid[q];
        int m;
        u16 *seg = segment(t, &m);
        int d = 1, pp = 0, prev;
        if (m <= 8) {
            // put in order by a network in registers, the padding to the end: one round trip to shared memory
            int v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = j < m ? seg[j] : 0x10000;
            sort_eight(v);
            prev = v[0];
            seg[0] = (u16)prev;
#pragma unroll
            for (int a = 1; a < 8; ++a) {
                const int x = v[a];
                if (a < m && x != prev) { if (x - prev >= 2) ++pp; seg[d++] = (u16)x; prev = x; }
            }
        } else {
            // (the scatter took the events nearly in order: hardly anything moves)
            for (int a = 1; a < m; ++a) {
                const u16 x = seg[a];
                int c = a - 1;
                while (c >= 0 && seg[c] > x) { seg[c + 1] = seg[c]; --c; }
                seg[c + 1] = x;
            }
            prev = seg[0];
            for (int a = 1; a < m; ++a) {
                const int x = seg[a];
                if (x != prev) { if (x - prev >= 2) ++pp; seg[d++] = (u16)x; prev = x; }
            }
        }
        dp[t] = (unsigned)d | (unsigned)pp << 16;
    }
    for (int q = warp; q < nheavy; q += kSmWarps) {
        const int t = s_mid[E - 1 - q];
        int m;
        u16 *seg = segment(t, &m);
        if (m > kSmWarpSort) continue;
        bitonic_sort<false>(seg, m, lane, 32);
        const unsigned r = small_compact_warp(seg, m, lane);
        if (lane == 0) dp[t] = r;
    }
    for (int q = 0; q < nheavy; ++q) {              // (the few that a block sorts better)
        const int t = s_mid[E - 1 - q];
        int m;
        u16 *seg = segment(t, &m);
        if (m <= kSmWarpSort) continue;
        bitonic_sort<true>(seg, m, tid, kSmThreads);
        if (warp == 0) { const unsigned r = small_compact_warp(seg, m, lane); if (lane == 0) dp[t] = r; }
    }
    __syncthreads();
    // (the sizes of the first tensors are on their way meanwhile)
    constexpr int kBook = 4;
    long long size[kBook];
    bool global[kBook];
    auto load_size = [&](int t00) {
#pragma unroll
        for (int q = 0; q < kBook; ++q) {
            const int t = t00 + q * kSmThreads + tid;
            size[q] = t < N ? A.t.tensor_bytes[t] : 1;
            global[q] = t < N && A.t.tensor_global != nullptr && A.t.tensor_global[t] != 0;
        }
    };
    if (clock) load_size(0);
    // ---- offsets of every tensor's uses and periods (16 bits each: both sums are at most E)
    const unsigned total = small_prefix<unsigned>(dp, N, s_w32);
    if (tid == 0) dp[N] = total;
    __syncthreads();
    const int D = (int)(total & 0xffffu), PC = (int)(total >> 16);
    const VitalityBuffers &out = A.v;
    bad = 0;
    if (D > out.uses_cap) bad |= G10_DEV_USES_OVERFLOW;
    if (PC > out.periods_cap) bad |= G10_DEV_PERIODS_OVERFLOW;
    const int raw = none ? 0 : (int)off[N - 1];
    const bool dense = D == raw;                    // no repeats: ks is the use list as it stands
    u16 *s_pos = s_id, *s_ten = s_krel;             // of every period: where its first use stands in ks, its tensor
    constexpr int kOut = 3;                         // tensors of a thread whose tables are read together
    for (int t0 = tid; t0 < N; t0 += kOut * kSmThreads) {
        unsigned x[kOut], y[kOut];
        int o[kOut], f[kOut], la[kOut];
#pragma unroll
        for (int q = 0; q < kOut; ++q) {
            const int t = t0 + q * kSmThreads;
            const bool in = t < N;
            x[q] = in ? dp[t] : 0u; y[q] = in ? dp[t + 1] : 0u;
            o[q] = in && t > 0 ? (int)off[t - 1] : 0;
        }
#pragma unroll
        for (int q = 0; q < kOut; ++q) {
            const int d = (int)((y[q] - x[q]) & 0xffffu);
            f[q] = d > 0 ? (int)ks[o[q]] : -1; la[q] = d > 0 ? (int)ks[o[q] + d - 1] : -1;
        }
#pragma unroll
        for (int q = 0; q < kOut; ++q) {
            const int t = t0 + q * kSmThreads;
            if (t >= N) break;
            const int d = (int)((y[q] - x[q]) & 0xffffu), uo = (int)(x[q] & 0xffffu), p0 = (int)(x[q] >> 16);
            out.first_use[t] = f[q]; out.last_use[t] = la[q]; out.num_uses[t] = d;
            out.use_ptr[t] = uo; out.period_ptr[t] = p0;
            if (!dense) for (int a = 0; a < d && uo + a < out.uses_cap; ++a) out.uses[uo + a] = ks[o[q] + a];
            if (y[q] >> 16 == (unsigned)p0) continue;         // (no period: nearly all)
            int po = p0, prev = f[q];
            for (int a = 1; a < d; ++a) {
                const int v = ks[o[q] + a];
                if (v - prev >= 2) { s_pos[po] = (u16)(o[q] + a - 1); s_ten[po] = (u16)t; ++po; }
                prev = v;
            }
        }
    }
    if (tid == 0) { out.use_ptr[N] = D; out.period_ptr[N] = PC; out.counts[0] = D; out.counts[1] = PC; }
    if (dense)
        for (int j = tid; j < D && j < out.uses_cap; j += kSmThreads) out.uses[j] = ks[j];
    __syncthreads();
#pragma unroll 4
    for (int p = tid; p < PC; p += kSmThreads) {
        const int i = s_pos[p];
        if (p < out.periods_cap) { out.period_tensor[p] = s_ten[p]; out.period_prev_use[p] = ks[i]; out.period_next_use[p] = ks[i + 1]; }
    }
    if (clock) {
        __syncthreads();
        // ---- pressure: sizes where the tensors are born and where they die, prefix sum, peak and its lowest slot
        long long everywhere = 0;                   // bytes of the global tensors
        int wrap_base = PC;
        for (int k = tid; k <= K; k += kSmThreads) s_diff[k] = 0;
        __syncthreads();
        for (int t00 = 0; t00 < N; t00 += kBook * kSmThreads) {
            if (t00 != 0) load_size(t00);
#pragma unroll
            for (int q = 0; q < kBook; ++q) {
                const int t = t00 + q * kSmThreads + tid;
                if (t00 + q * kSmThreads >= N) break;
                const long long b = size[q];
                bool wrap = false;
                int f = 0, la = 0;
                if (t < N) {
                    int m;
                    const u16 *seg = segment(t, &m);
                    const int d = (int)((dp[t + 1] - dp[t]) & 0xffffu);
                    if (b < 1 || b >= ((long long)1 << 40)) bad |= G10_DEV_BAD_BYTES;
                    if (d > 0) {
                        f = seg[0]; la = seg[d - 1];
                        if (global[q]) { everywhere += b; wrap = f + K - la >= 2; }
                        else { small_add64(&s_diff[f], b); small_add64(&s_diff[la + 1], -b); }
                    }
                }
                if (A.start2 != nullptr) {
                    // steady state: the period of a global tensor that spans two iterations, behind the ordinary ones in tensor order
                    unsigned n;
                    const unsigned at = small_scan<unsigned>(wrap ? 1u : 0u, s_w32, &n);
                    const int64_t p = (int64_t)wrap_base + at;
                    if (wrap) {
                        if (p < out.periods_cap) { out.period_tensor[p] = t; out.period_prev_use[p] = la; out.period_next_use[p] = f + K; }
                        else bad |= G10_DEV_PERIODS_OVERFLOW;
                    }
                    wrap_base += (int)n;
                }
            }
        }
        if (A.start2 != nullptr && tid == 0) out.counts[1] = wrap_base;
        everywhere = warp_sum_i64(everywhere);
        if (lane == 0 && everywhere != 0) small_add64(&s_diff[0], everywhere);
        __syncthreads();
        const int c = ((K + kSmThreads - 1) / kSmThreads) | 1, lo = tid * c < K ? tid * c : K, hi = lo + c < K ? lo + c : K;
        long long sum = 0, all, mx = 0;
        int sl = -1;
#pragma unroll 4
        for (int k = lo; k < hi; ++k) sum += s_diff[k];
        long long run = small_scan<long long>(sum, s_w64, &all);
#pragma unroll 4
        for (int k = lo; k < hi; ++k) {
            run += s_diff[k];
            s_diff[k] = run;
            if (sl < 0 || run > mx) { mx = run; sl = k; }
        }
        small_peak(mx, sl);
        __syncthreads();
        if (lane == 0) { s_w64[warp] = mx; s_sl[warp] = sl; }
#pragma unroll 4
        for (int k = tid; k < K; k += kSmThreads) A.pressure[k] = s_diff[k];
        __syncthreads();
        if (warp == 0) {
            mx = s_w64[lane]; sl = s_sl[lane];
            small_peak(mx, sl);
            if (lane == 0) { *A.peak_bytes = mx; *A.peak_slot = sl; }
        }
    }
    {
        const unsigned w = __reduce_or_sync(0xffffffffu, bad);
        if (lane == 0 && w) atomicOr(&s_bits, w);
    }
    __syncthreads();
    if (tid == 0) {
        const int64_t st = (int64_t)s_bits;
        if (A.status_counts != nullptr) *A.status_counts = st;
        if (A.status_timeline != nullptr) *A.status_timeline = st;
        if (A.status_word != nullptr) *A.status_word = (ull)st;
        if (A.done != nullptr) *A.done = 0u;
    }
}

static size_t small_budget()
{
    static int known[kMaxDevices];
    return (size_t)dynamic_smem_room((const void *)k_small, known);
}

// This kernel for whatever fits it.  Measured against the general passes (us, whole calls; trace on the device: here / there, in
// pinned host memory: here / there): 96 kernels and 320 events 13 / 28, 30 / 58; 1652 and 5268: 18.5 / 36.9, 38 / 69; 3346 and 12 600:
// 26.7 / 40.0, 49 / 77; 6692 and 25 200 (7721 tensors): 43.1 / 50.6, 77 / 95.  With many tensors of few uses the general passes draw level
// on the device, and only there: 2000 kernels, 8000 tensors, 9860 events 24.6 / 39.5, 48 / 77; 3000, 12 000, 14 819: 32.8 / 32.0, 59 / 72;
// 6000, 12 000, 14 891: 36.9 / 33.1, 70 / 77; 7000, 10 500, 13 047: 35.8 / 34.9, 69 / 77.  What a line below the shared memory's end could
// give is a tenth on a few device traces between 12 000 tensors and that end.
bool small_analysis_fits(int64_t K, int64_t N, int64_t E)
{
    if (K < 1 || N < 1 || E < 1 || K >= 65535 || N >= 65535 || E >= 65535) return false;
    return small_layout(K, N, E).total <= small_budget();
}

cudaError_t launch_small(const SmallArgs &A, cudaStream_t s)
{
    const size_t smem = small_layout(A.t.K, A.t.N, A.t.E).total;
    if (const cudaError_t e = allow_launch((const void *)k_small, small_budget(), 1); e != cudaSuccess) return e;
    k_small<<<1, kSmThreads, smem, s>>>(A); count_launch();
    return cudaGetLastError();
}

}  // namespace g10
