// Code instrumentation (Section 4.4, Figure 9): the stream of g10_alloc / g10_free / g10_pre_evict /
// g10_prefetch calls, ordered by kernel boundary, then FREE < PRE_EVICT < ALLOC < PREFETCH, then tensor id.
//
// Every instruction is one 64-bit key (boundary << 33 | opcode << 31 | tensor; unique) plus the plan record it
// came from.  The keys are sorted with the same shape as the vitality pass: boundaries are cut into buckets of
// consecutive boundaries holding a couple of thousand instructions, a histogram sizes the buckets -- kept per block of
// the counting kernel, so that the scatter kernel, whose blocks walk the same items, knows each block's own run inside
// every bucket and places its keys with shared-memory counters alone (no global cursor) --, the keys are
// scattered into their bucket's slice, and one block per bucket sorts its slice in shared memory (counting sort by
// boundary, then the few instructions of every boundary in key order by one thread; a boundary with more than 32
// by a bitonic network), which also gives the CSR pointers, and writes the records out in order.
// A bucket too large for shared memory (very many tensors allocated at one boundary) is sorted in global memory.
#include "g10_device.cuh"
#include "g10_internal.h"
#include <cstddef>

namespace g10 {

constexpr int kEmitThreads = 512;
constexpr int kEmitCap = 4096;            // instructions of a bucket sorted in shared memory
enum { kOpFree = 0, kOpPreEvict = 1, kOpAlloc = 2, kOpPrefetch = 3 };

struct EmitArgs {
    int64_t K, N, n;
    const int32_t *first_use, *last_use;
    const int64_t *bytes;
    const uint8_t *glob;
    const int64_t *start;
    const g10_migration *mig;
    const int64_t *new_issue;
    int bw, nb;                           // boundaries per bucket, buckets
    ull magic;                            // ceil(2^64 / bw) (0 when bw == 1): the bucket of boundary x is the high half of x * magic
    unsigned *bucket_count, *bucket_cursor;
    unsigned *block_count;                // [G][nb] what each block of the counting kernel saw of every bucket, then the running sums
    int G;                                // blocks of the counting and of the scatter kernel (the same items go to the same block)
    ull *keys;
    int32_t *payload;
    unsigned *ticket;
    ull *status;
};

// A pre-eviction (item < n) or a prefetch of a plan record -> boundary, opcode, record
__device__ __forceinline__ void emit_record(const EmitArgs &A, int64_t item, int64_t *boundary, int *opcode, int *record)
{
    const bool evict = item < A.n;
    const int64_t r = evict ? item : item - A.n;
    int64_t t = evict ? A.mig[r].evict_issue_ns : (A.new_issue ? A.new_issue[r] : A.mig[r].prefetch_issue_ns);
    // (a steady-state plan: the prefetch of a wrap-around period may lie in the next iteration; it stands at the same
    // moment of this one)
    if (!evict && t >= A.start[A.K]) t -= A.start[A.K];
    // last boundary b in [0, K] with start[b] <= t (for a pre-eviction start[b] == t_r exactly).  Seven probes a step, all on their
    // way together: a third of the round trips of a binary search
    int lo = 0, hi = (int)A.K;
    while (lo < hi) {
        const int step = (hi - lo) / 8 + 1;
        int c = 0;
#pragma unroll
        for (int j = 1; j < 8; ++j) { const int64_t x = (int64_t)lo + (int64_t)j * step; c += x <= hi && A.start[x <= hi ? x : hi] <= t ? 1 : 0; }
        lo += c * step;
        if (c < 7 && lo + step - 1 < hi) hi = lo + step - 1;
    }
    *boundary = lo; *opcode = evict ? kOpPreEvict : kOpPrefetch; *record = (int)r;
}

// Calls put(valid, boundary, opcode, tensor, record), whole warps at a time, for the instructions of the block's share of the work:
// the plan's records (first: their searches take longest), then every tensor's allocation and release.  The same items go to the
// same block in every kernel.
template <typename F>
__device__ __forceinline__ void emit_items(const EmitArgs &A, F &&put)
{
    constexpr int kBatch = 4;                 // tensors a thread reads together
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * kEmitThreads, total = 2 * A.n + A.N;
    for (int64_t w0 = (int64_t)blockIdx.x * kEmitThreads + (threadIdx.x - lane); w0 < total; w0 += kBatch * stride) {
        int f[kBatch], la[kBatch];
        bool g[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int64_t i = w0 + lane + u * stride - 2 * A.n;
            const bool in = i >= 0 && i < A.N;
            f[u] = in ? A.first_use[i] : -1;
            la[u] = in ? A.last_use[i] : 0;
            g[u] = in && A.glob != nullptr && A.glob[i] != 0;
        }
#pragma unroll 1
        for (int64_t r0 = w0; r0 < 2 * A.n && r0 < w0 + kBatch * stride; r0 += stride) {
            int64_t bd = 0;
            int op = 0, rc = -1, tn = 0;
            const bool in = r0 + lane < 2 * A.n;
            if (in) { emit_record(A, r0 + lane, &bd, &op, &rc); tn = A.mig[rc].tensor; }
            put(in, bd, op, tn, rc);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (w0 + u * stride >= total) break;
            const int i = (int)(w0 + lane + u * stride - 2 * A.n);
            put(f[u] >= 0, (int64_t)(g[u] ? 0 : f[u]), (int)kOpAlloc, i, -1);
            put(f[u] >= 0 && !g[u], (int64_t)la[u] + 1, (int)kOpFree, i, -1);
        }
    }
}

// The next free place of every lane's bucket (shared-memory counters).  Neighbouring tensors are born and die at neighbouring
// kernels: most lanes of a warp want the same bucket, and one lane counts for those that want the first one's (32 atomics on one
// word take turns; sorting out all of a warp's buckets with match.any took as long).
__device__ __forceinline__ unsigned emit_take(unsigned *next, bool valid, int b)
{
    const int lane = threadIdx.x & 31;
    const unsigned on = __ballot_sync(0xffffffffu, valid);
    if (on == 0u) return 0u;
    const int first = __ffs(on) - 1, b0 = __shfl_sync(0xffffffffu, b, first);
    const unsigned same = __ballot_sync(0xffffffffu, valid && b == b0);
    unsigned at = 0;
    if (lane == first) at = atomicAdd(&next[b0], (unsigned)__popc(same));
    else if (valid && b != b0) at = atomicAdd(&next[b], 1u);
    const unsigned run = __shfl_sync(0xffffffffu, at, first) + __popc(same & ((1u << lane) - 1u));
    return b == b0 ? run : at;
}

// Bucket of a boundary.  With magic = (2^64 + e) / bw, 0 <= e < bw, the product x * magic / 2^64 exceeds x / bw by less than
// 2^-32 for x < 2^32, and x / bw is at least 1 / bw short of the next integer: the high half is the quotient exactly.
__device__ __forceinline__ int emit_bucket(const EmitArgs &A, int64_t boundary)
{
    return A.magic ? (int)__umul64hi((ull)boundary, A.magic) : (int)boundary;
}

__device__ __forceinline__ ull emit_key(int64_t boundary, int opcode, int tensor)
{
    return ((ull)boundary << 33) | ((ull)opcode << 31) | (ull)(unsigned)tensor;
}

__global__ void __launch_bounds__(kEmitThreads) k_emit_hist(EmitArgs A)
{
    extern __shared__ unsigned s_hist[];
    for (int b = threadIdx.x; b < A.nb; b += kEmitThreads) s_hist[b] = 0;
    __syncthreads();
    emit_items(A, [&](bool valid, int64_t bd, int, int, int) { emit_take(s_hist, valid, emit_bucket(A, bd)); });
    __syncthreads();
    // what this block saw of every bucket: the scatter kernel, whose blocks walk the same items, gets from it the block's own
    // run inside every bucket's slice and needs no global cursor
    for (int b = threadIdx.x; b < A.nb; b += kEmitThreads) A.block_count[(size_t)blockIdx.x * A.nb + b] = s_hist[b];
}

// Per bucket: running sums over the blocks (in place) and the bucket's total.  A block takes 8 buckets (a sector of every row) and has
// 128 threads for each, which split the counting blocks among them (32 buckets a block and 32 threads each: 7.5 us instead of 5).
constexpr int kOffThreads = 1024, kOffBuckets = 8, kOffRows = (kEmitMaxBlocks * kOffBuckets + kOffThreads - 1) / kOffThreads;
__global__ void __launch_bounds__(kOffThreads) k_emit_block_offsets(EmitArgs A)
{
    __shared__ unsigned s_sum[kOffThreads / 32][kOffBuckets];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, at = threadIdx.x % kOffBuckets, b = blockIdx.x * kOffBuckets + at;
    const int groups = kOffThreads / kOffBuckets, rows = (A.G + groups - 1) / groups, r0 = threadIdx.x / kOffBuckets * rows;       // (rows <= kOffRows)
    unsigned v[kOffRows], sum = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
    for (int q = 0; q < kOffRows; ++q) { v[q] = q < rows && r0 + q < A.G && b < A.nb ? A.block_count[(size_t)(r0 + q) * A.nb + b] : 0u; sum += v[q]; }
    unsigned incl = sum;
#pragma unroll
    for (int o = kOffBuckets; o < 32; o <<= 1) { const unsigned y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
    if (lane >= 32 - kOffBuckets) s_sum[warp][at] = incl;
    __syncthreads();
    unsigned run = incl - sum, all = 0;
#pragma unroll
    for (int x = 0; x < kOffThreads / 32; ++x) { const unsigned y = s_sum[x][at]; if (x < warp) run += y; all += y; }
    if (b >= A.nb) return;
#pragma unroll
    for (int q = 0; q < kOffRows; ++q) if (q < rows && r0 + q < A.G) { A.block_count[(size_t)(r0 + q) * A.nb + b] = run; run += v[q]; }
    if (threadIdx.x < kOffBuckets) A.bucket_count[b] = all;
}

// exclusive scan of the bucket counts (nb <= 4096) into s_base[0..nb]
__device__ __forceinline__ void emit_scan_buckets(const unsigned *cnt, int nb, long long *s_base, long long *s_w)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long carry = 0;
    for (int base = 0; base < nb; base += kEmitThreads) {
        const int j = base + threadIdx.x;
        const long long v = j < nb ? (long long)cnt[j] : 0;
        const long long incl = warp_inclusive_scan_i64(v, lane);
        __syncthreads();
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        long long wpre = 0, tot = 0;
        for (int w = 0; w < kEmitThreads / 32; ++w) { const long long x = s_w[w]; if (w < warp) wpre += x; tot += x; }
        if (j < nb) s_base[j] = carry + wpre + incl - v;
        carry += tot;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_base[nb] = carry;
    __syncthreads();
}

__global__ void __launch_bounds__(kEmitThreads) k_emit_scatter(EmitArgs A)
{
    extern __shared__ long long s_base[];            // [nb + 1] first slot of each bucket, then [nb] (unsigned) this block's next slot inside it
    __shared__ long long s_w[kEmitThreads / 32];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    emit_scan_buckets(A.bucket_count, A.nb, s_base, s_w);
    unsigned *s_next = (unsigned *)(s_base + A.nb + 1);
    for (int b = threadIdx.x; b < A.nb; b += kEmitThreads) s_next[b] = A.block_count[(size_t)blockIdx.x * A.nb + b];
    __syncthreads();
    emit_items(A, [&](bool valid, int64_t bd, int op, int tn, int rc) {
        const int b = emit_bucket(A, bd);
        const unsigned at = emit_take(s_next, valid, b);                   // (shared memory: the block's own run of the bucket)
        if (!valid) return;
        const long long pos = s_base[b] + at;
        A.keys[pos] = emit_key(bd, op, tn);
        if (rc >= 0) A.payload[pos] = rc;          // (only the few instructions that come from a plan record carry one: the
                                                   // others' payload is never read, which spares a scattered store per tensor)
    });
}

// bitonic network over (key, payload) pairs; arbitrary n (values only ever move up)
__device__ void emit_bitonic(ull *k, int32_t *p, int n)
{
    int n2 = 1;
    while (n2 < n) n2 <<= 1;
    for (int kk = 2; kk <= n2; kk <<= 1) {
        for (int j = kk >> 1, lj = 31 - __clz(kk >> 1); j > 0; j >>= 1, --lj) {
            const bool mirror = (j == (kk >> 1));
            for (int t = threadIdx.x; t < n2 / 2; t += blockDim.x) {
                const int blk = t >> lj, off = t & (j - 1);
                const int i = blk * 2 * j + off;
                const int q = mirror ? (blk * 2 * j + 2 * j - 1 - off) : (i + j);
                if (q < n) {
                    const ull x = k[i], y = k[q];
                    if (x > y) { k[i] = y; k[q] = x; const int32_t px = p[i]; p[i] = p[q]; p[q] = px; }
                }
            }
            __syncthreads();
        }
    }
}

static_assert(sizeof(g10_instruction) == 32 && offsetof(g10_instruction, opcode) == 0 && offsetof(g10_instruction, tensor) == 4 &&
              offsetof(g10_instruction, target) == 8 && offsetof(g10_instruction, record) == 12 && offsetof(g10_instruction, bytes) == 16 &&
              offsetof(g10_instruction, time_ns) == 24, "k_emit_write assembles the record from four 64-bit words");
constexpr int kEmitStageStride = 36;      // (32 + 4: the four word planes of a warp's tile fall into different banks)
constexpr int kEmitRegs = kEmitCap / kEmitThreads;   // keys a thread keeps in registers between the two passes
constexpr int kEmitWide = 32;                        // a boundary with more instructions is sorted by the whole block

__global__ void __launch_bounds__(kEmitThreads, 2) k_emit_write(EmitArgs A, int64_t *inst_ptr, g10_instruction *inst, int64_t inst_cap, int64_t *counts)
{
    extern __shared__ long long s_dyn[];
    long long *s_base = s_dyn;                                   // [nb + 1]
    int *s_cnt = (int *)(s_base + A.nb + 1);                     // [bw + 1] instructions per boundary of the bucket, then their offsets
    int *s_cur = s_cnt + A.bw + 1;                               // [bw] fill cursors
    ull *s_keys = (ull *)(((uintptr_t)(s_cur + A.bw) + 7) & ~(uintptr_t)7);               // [kEmitCap]
    int32_t *s_pay = (int32_t *)(s_keys + kEmitCap);              // [kEmitCap]
    ull *s_stage = (ull *)(s_pay + kEmitCap);                     // [warps][4][kEmitStageStride] the records of a warp on their way out
    __shared__ long long s_w[kEmitThreads / 32];
    __shared__ int s_bucket, s_nwide;
    __shared__ int s_wide[64];
    const int bw = A.bw;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    emit_scan_buckets(A.bucket_count, A.nb, s_base, s_w);
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) { s_bucket = (int)atomicAdd(A.ticket, 1u); s_nwide = 0; }
        __syncthreads();
        const int b = s_bucket;
        if (b >= A.nb) break;
        const long long base = s_base[b];
        const int n = (int)(s_base[b + 1] - base);
        ull *gk = A.keys + base;
        int32_t *gp = A.payload + base;
        const int64_t b0 = (int64_t)b * bw;
        const int bw_eff = (int)((A.K + 1 - b0) < bw ? (A.K + 1 - b0) : bw);
        for (int j = threadIdx.x; j <= bw_eff; j += kEmitThreads) { s_cnt[j] = 0; if (j < bw_eff) s_cur[j] = 0; }
        __syncthreads();
        const ull *kp; const int32_t *pp;
        if (n <= kEmitCap) {
            // Counting sort by boundary in shared memory (the keys stay in registers between the two passes), then
            // every boundary's few instructions are put in key order by one thread; the keys are unique, so this is
            // the order a sort of the whole bucket would give.
            ull rk[kEmitRegs];
#pragma unroll
            for (int q = 0; q < kEmitRegs; ++q) {
                const int j = q * kEmitThreads + threadIdx.x;
                rk[q] = j < n ? gk[j] : ~0ull;
            }
#pragma unroll
            for (int q = 0; q < kEmitRegs; ++q)
                if (rk[q] != ~0ull) atomicAdd(&s_cnt[(int)((rk[q] >> 33) - b0)], 1);
            __syncthreads();
            {   // in-place exclusive scan of s_cnt[0..bw_eff), total in s_cnt[bw_eff]
                const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
                int carry = 0;
                for (int c0 = 0; c0 < bw_eff; c0 += kEmitThreads) {
                    const int j = c0 + threadIdx.x;
                    const int v = j < bw_eff ? s_cnt[j] : 0;
                    int incl = v;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
                    __syncthreads();
                    if (lane == 31) s_w[warp] = incl;
                    __syncthreads();
                    int wpre = 0, tot = 0;
                    for (int w = 0; w < kEmitThreads / 32; ++w) { const int x = (int)s_w[w]; if (w < warp) wpre += x; tot += x; }
                    if (j < bw_eff) s_cnt[j] = carry + wpre + incl - v;
                    carry += tot;
                }
                __syncthreads();
                if (threadIdx.x == 0) s_cnt[bw_eff] = carry;
                __syncthreads();
            }
#pragma unroll
            for (int q = 0; q < kEmitRegs; ++q)
                if (rk[q] != ~0ull) {
                    const int j = q * kEmitThreads + threadIdx.x;
                    const int bd = (int)((rk[q] >> 33) - b0);
                    const int slot = s_cnt[bd] + atomicAdd(&s_cur[bd], 1);
                    s_keys[slot] = rk[q];
                    s_pay[slot] = ((rk[q] >> 31) & 1u) ? gp[j] : -1;       // (PRE_EVICT = 1 and PREFETCH = 3 come from a plan record)
                }
            __syncthreads();
            // Inside a boundary the keys go in key order.  Every thread takes back the instructions at its slots, finds for
            // each its rank among the instructions of its boundary by counting the smaller keys (a boundary holds a handful;
            // keys are unique, so ranks are too), and puts it where it belongs.  One thread sorting one boundary, as before,
            // makes the whole block wait for the boundary with the most instructions.
            {
                ull ik[kEmitRegs];
                int ip[kEmitRegs], dst[kEmitRegs];
#pragma unroll
                for (int q = 0; q < kEmitRegs; ++q) {
                    const int j = q * kEmitThreads + threadIdx.x;
                    dst[q] = -1;
                    if (j < n) {
                        ik[q] = s_keys[j]; ip[q] = s_pay[j];
                        const int bd = (int)((ik[q] >> 33) - b0);
                        const int o = s_cnt[bd], m = s_cnt[bd + 1] - o;
                        if (m <= kEmitWide) {
                            int r = 0;
                            for (int a = 0; a < m; ++a) r += s_keys[o + a] < ik[q] ? 1 : 0;
                            dst[q] = o + r;
                        } else if (j == o) { const int w2 = atomicAdd(&s_nwide, 1); if (w2 < 64) s_wide[w2] = bd; }   // (its first slot reports it)
                    }
                }
                __syncthreads();
#pragma unroll
                for (int q = 0; q < kEmitRegs; ++q)
                    if (dst[q] >= 0) { s_keys[dst[q]] = ik[q]; s_pay[dst[q]] = ip[q]; }
            }
            __syncthreads();
            const int nwide = s_nwide;
            for (int hq = 0; hq < (nwide <= 64 ? nwide : bw_eff); ++hq) {
                const int bd = nwide <= 64 ? s_wide[hq] : hq;
                const int o = s_cnt[bd], m = s_cnt[bd + 1] - o;
                if (m <= kEmitWide) continue;                      // (only when the list overflowed: uniform test)
                emit_bitonic(s_keys + o, s_pay + o, m);
            }
            kp = s_keys; pp = s_pay;
        } else {
            emit_bitonic(gk, gp, n);
            for (int j = threadIdx.x; j < n; j += kEmitThreads) atomicAdd(&s_cnt[(int)((gk[j] >> 33) - b0)], 1);
            __syncthreads();
            {   // in-place exclusive scan of s_cnt[0..bw_eff)
                const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
                int carry = 0;
                for (int c0 = 0; c0 < bw_eff; c0 += kEmitThreads) {
                    const int j = c0 + threadIdx.x;
                    const int v = j < bw_eff ? s_cnt[j] : 0;
                    int incl = v;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
                    __syncthreads();
                    if (lane == 31) s_w[warp] = incl;
                    __syncthreads();
                    int wpre = 0, tot = 0;
                    for (int w = 0; w < kEmitThreads / 32; ++w) { const int x = (int)s_w[w]; if (w < warp) wpre += x; tot += x; }
                    if (j < bw_eff) s_cnt[j] = carry + wpre + incl - v;
                    carry += tot;
                }
                __syncthreads();
            }
            kp = gk; pp = gp;
        }
        // CSR pointers of the bucket's boundaries
        for (int j = threadIdx.x; j < bw_eff; j += kEmitThreads) inst_ptr[b0 + j] = base + s_cnt[j];
        if (b == A.nb - 1 && threadIdx.x == 0) {
            inst_ptr[A.K + 1] = s_base[A.nb];
            counts[0] = s_base[A.nb];
            if (s_base[A.nb] > inst_cap) raise_status(A.status, G10_DEV_PLAN_OVERFLOW);
        }
        // the records, in order.  A thread that stored its own 32-byte record would write every 32-byte sector in four pieces
        // (four 8-byte stores at a stride of 32 bytes across the warp); the 32 records of a warp go through a small
        // shared-memory tile instead and leave as four contiguous 256-byte runs.
        {
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            ull *st = s_stage + warp * (4 * kEmitStageStride);
            constexpr int kBatch = 4;                                      // rounds whose sizes and times are read together
            for (int j1 = 0; j1 < n; j1 += kBatch * kEmitThreads) {
                ull size[kBatch];
                int64_t when[kBatch];
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    const int j = j1 + u * kEmitThreads + threadIdx.x;
                    const bool in = j < n && base + j < inst_cap;
                    const ull key = in ? kp[j] : 0;
                    size[u] = in ? (ull)A.bytes[key & 0x7fffffffu] : 0;
                    when[u] = in ? A.start[key >> 33] : 0;
                }
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    const int j0 = j1 + u * kEmitThreads, j = j0 + threadIdx.x;
                    if (j0 >= n) break;
                    ull w0 = 0, w1 = 0, w2 = 0, w3 = 0;
                    if (j < n && base + j < inst_cap) {
                        const ull key = kp[j];
                        const int opcode = (int)((key >> 31) & 3u), tensor = (int)(key & 0x7fffffffu), record = (opcode & 1) ? pp[j] : -1;
                        int target = -1;
                        int64_t time_ns = when[u];
                        if (opcode == kOpPreEvict) { target = A.mig[record].dest; time_ns = A.mig[record].evict_issue_ns; }
                        if (opcode == kOpPrefetch) {
                            time_ns = A.new_issue ? A.new_issue[record] : A.mig[record].prefetch_issue_ns;
                            if (time_ns >= A.start[A.K]) time_ns -= A.start[A.K];      // (steady-state plans: see emit_record)
                        }
                        w0 = (ull)(unsigned)opcode | ((ull)(unsigned)tensor << 32);
                        w1 = (ull)(unsigned)target | ((ull)(unsigned)record << 32);
                        w2 = size[u];
                        w3 = (ull)time_ns;
                    }
                    st[0 * kEmitStageStride + lane] = w0; st[1 * kEmitStageStride + lane] = w1;
                    st[2 * kEmitStageStride + lane] = w2; st[3 * kEmitStageStride + lane] = w3;
                    __syncwarp();
                    const long long first = base + j0 + warp * 32;              // the warp's first record
                    long long nrec = n - (j0 + warp * 32);
                    if (inst_cap - first < nrec) nrec = inst_cap - first;
                    if (nrec > 32) nrec = 32;
                    ull *dst = reinterpret_cast<ull *>(inst + first);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int i = q * 32 + lane;                          // 8-byte word of the warp's 1024 bytes
                        if ((i >> 2) < nrec) dst[i] = st[(i & 3) * kEmitStageStride + (i >> 2)];
                    }
                    __syncwarp();
                }
            }
        }
    }
}

bool emit_choose_buckets(int64_t K, int64_t total_items, int sms, int *bw, int *nb, ull *magic)
{
    // boundaries per bucket so that a bucket holds about 3000 instructions (kEmitCap = 4096 are sorted in shared memory; a
    // fuller bucket goes the slow way); at most 4096 buckets of 4096 boundaries.  k_emit_write takes the buckets one per block
    // at a time with two blocks per SM: with more buckets than blocks they are narrowed to whole rounds of its grid (sms > 0).
    const int64_t B = K + 1;
    int64_t w = total_items > 0 ? (3000 * B) / total_items : 4096;
    w = w < 1 ? 1 : (w > 4096 ? 4096 : w);
    int64_t buckets = (B + w - 1) / w;
    if (buckets > 4096) { w = (B + 4095) / 4096; buckets = (B + w - 1) / w; }
    if (w > 4096) return false;
    const int64_t G = 2 * (int64_t)sms;
    if (G > 0 && buckets > G) {
        const int64_t target = (buckets + G - 1) / G * G;
        if (target <= 4096) { w = (B + target - 1) / target; buckets = (B + w - 1) / w; }
    }
    *bw = (int)w; *nb = (int)buckets;
    *magic = w == 1 ? 0 : ~(ull)0 / (ull)w + 1;
    return true;
}

cudaError_t launch_emit(const EmitLaunch &L, cudaStream_t s)
{
    EmitArgs A;
    A.K = L.K; A.N = L.N; A.n = L.n;
    A.first_use = L.first_use; A.last_use = L.last_use; A.bytes = L.bytes; A.glob = L.glob; A.start = L.start;
    A.mig = L.mig; A.new_issue = L.new_issue;
    A.bucket_count = L.bucket_count; A.bucket_cursor = L.bucket_cursor; A.keys = L.keys; A.payload = L.payload;
    A.ticket = L.ticket; A.status = L.status;
    const int sms = current_sm_count();
    if (sms <= 0) return cudaErrorInvalidDevice;
    if (!emit_choose_buckets(L.K, 2 * L.N + 2 * L.n, sms, &A.bw, &A.nb, &A.magic)) return cudaErrorInvalidValue;
    const int64_t total = L.N + 2 * L.n;
    int64_t g = (total + kEmitThreads - 1) / kEmitThreads;
    if (g > 4 * (int64_t)sms) g = 4 * (int64_t)sms;
    if (g > kEmitMaxBlocks) g = kEmitMaxBlocks;
    if (g < 1) g = 1;
    A.block_count = L.block_count; A.G = (int)g;
    k_emit_hist<<<(int)g, kEmitThreads, sizeof(unsigned) * (size_t)A.nb, s>>>(A); count_launch();
    // (the kernels behind the first are placed while their predecessor drains; they wait for it themselves)
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s; cfg.attrs = attr; cfg.numAttrs = 1;
    cfg.gridDim = dim3((A.nb + kOffBuckets - 1) / kOffBuckets); cfg.blockDim = dim3(kOffThreads);
    cudaError_t e1 = cudaLaunchKernelEx(&cfg, k_emit_block_offsets, A);
    if (e1 != cudaSuccess) return e1;
    cfg.blockDim = dim3(kEmitThreads);
    const size_t sm2 = sizeof(long long) * (size_t)(A.nb + 1) + sizeof(unsigned) * (size_t)A.nb;
    cudaError_t e2 = allow_any<k_emit_scatter>();
    if (e2 != cudaSuccess) return e2;
    cfg.gridDim = dim3((unsigned)g); cfg.dynamicSmemBytes = sm2;
    e1 = cudaLaunchKernelEx(&cfg, k_emit_scatter, A);
    if (e1 != cudaSuccess) return e1;
    const size_t sm3 = sizeof(long long) * (size_t)(A.nb + 1) + sizeof(int) * (size_t)(2 * A.bw + 2) + 8 +
                       (sizeof(ull) + sizeof(int32_t)) * kEmitCap + sizeof(ull) * (kEmitThreads / 32) * 4 * kEmitStageStride;
    cudaError_t e = allow_any<k_emit_write>();
    if (e != cudaSuccess) return e;
    const int g3 = A.nb < 2 * sms ? A.nb : 2 * sms;
    cfg.gridDim = dim3(g3); cfg.dynamicSmemBytes = sm3;
    e1 = cudaLaunchKernelEx(&cfg, k_emit_write, A, L.inst_ptr, L.inst, L.inst_cap, L.counts);
    return e1 != cudaSuccess ? e1 : cudaGetLastError();
}

}  // namespace g10
