// Algorithm 1 for traces whose timeline fits the shared memory of one SM (every DNN-shaped configuration): the greedy loop
// run by ONE thread-block cluster (one block is the smallest cluster), everything it touches in shared memory.
//
// Every block of the cluster holds its own copy of the timeline -- pressure above capacity and slot clock per slot, the
// smallest / largest value, a pending offset and a time stamp per tile of 32 slots, and per channel one bit "something is booked
// here" and one bit "full" per slot -- and owns every C-th inactive period.  A period carries its current destination, the benefit
// it had when it was last scored (an upper bound of the present one, because pressure only falls) and when that was.  The periods
// of a block lie in at most 32 groups with their best kept, so that one warp finds the block's best with one look.  One iteration:
//   S  warp 0 takes the best period by bound.  Its score is exact if no tile of its absent range has changed since it was scored
//      (or only tiles that are still at least the tensor's size above capacity throughout); else it is rescored from the tiles and
//      the warp looks again.  The block's best goes to all blocks of the cluster as asynchronous stores into their shared memory,
//      counted by a transaction barrier there; a bound that lies well below the last winner's score goes out as it is, and only if
//      it turns out in front is it made exact.
//   C  the winner is applied to every block's copy of the timeline: tiles wholly inside the absent range only change their offset,
//      the two tiles at its ends are rewritten; the transfer windows set bits, and one booked amount each.  Every thread compares
//      its periods' transfer windows with the winner's (one subtraction per pair of ranges); where they meet on the same channel, a
//      destination is lost if a slot it needs wholly has been booked, or if the one slot it needs in part has too little left.
//      Channels only fill up, so a destination that failed is out for good: SSD -> host (if its windows are free) -> erased.
// What bounds it: the instructions of one warp, one after the other, and the slowest of the blocks.  An iteration of the ResNet-152
// step takes 7.2 k cycles: 660 for the groups' best and a barrier, 1260-1550 for the search, 625 to send, 2600-2800 of waiting for
// the block that has to rescore, 1000 to decide, 810 to apply and check.  Outside the block barrier an instruction takes 7.7 cycles
// (2.5 fixed latency, 1.2 shared memory and reductions, 1.2 other loads and waits, 1.0 branches, 1.0 issue, 0.6 fetch); the exchange
// itself is 550-680 cycles.
//
// Scores are compared as rounded 64-bit ratios; candidates within kBand units in the last place of the best are told apart by
// the exact 128-bit cross products (lowest period index on ties).
//
// Batch mode (kBatch): one cluster per VARIANT of the same trace -- its own kernel durations, bandwidths and capacities.  A
// variant's blocks build their own slot clock (block-wide scan of its durations) and the geometry of their periods.
#include "g10_planner.cuh"

namespace g10 {

constexpr int kChipThreads = 256;
constexpr int kChipWarps = kChipThreads / 32;
constexpr int kChipMaxPeriods = 4096;        // per block (32 groups of at most 128)
// A key is the benefit (rounded to a double, at most twice) times the rounded inverse of the cost, rounded: at most 4 units in
// the last place off.  The exactly best candidate is therefore never more than 8 below the largest key.
constexpr ull kBand = 10;
constexpr int kAlone = 3;                    // periods warp 0 rescores in an iteration before it asks the other warps for help
static_assert(kAlone > 0, "with none, those asked for help would give up before their first, and be asked again");
constexpr unsigned kNoRange = 0xffffffffu;   // (destination unusable)

struct ChipArgs {
    unsigned *done;          // set to 1 when this kernel produced the plan
    int smem_bytes;          // dynamic shared memory the launch provides
    int64_t *busy_global;    // [cluster size][4][K], hocc_global [cluster size][K]: used when they do not fit shared memory
    int64_t *hocc_global;    // (null in batch mode: everything has to fit)
    int alone;               // the only planner of the call: works the geometry out itself and hands the status word over
};

// The best period of a block, as the blocks of the cluster tell each other.
struct __align__(16) ChipCand {
    ull key, ben_lo;
    ulonglong2 data;
    uint4 rec;               // eviction window | destination << 15, prefetch window, absent slots, bits 64.. of the benefit
};
static_assert(sizeof(ChipCand) == 48, "three 16-byte stores per block");
// What warp 0 tells the other warps.
enum { kFound, kNone, kHelp, kGaveUp };
struct __align__(16) ChipWinner {
    ChipCand c;
    int what, idx;           // period
};

// ---- thread-block clusters ---------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned cluster_rank() { unsigned r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ unsigned cluster_size() { unsigned r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned peer_addr(unsigned addr, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 16 bytes into a peer's shared memory, counted by a transaction barrier of that peer
__device__ __forceinline__ void st_async_v4(unsigned addr, uint4 v, unsigned bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(v.x), "r"(v.y),
                 "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void bar_init(unsigned bar, unsigned count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory"); }
__device__ __forceinline__ void bar_expect(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Waits until the phase with that parity is over; gives up after kBarrierTimeoutNs.
__device__ __forceinline__ bool bar_wait(unsigned bar, unsigned parity)
{
    ull t0 = 0;
    unsigned polls = 0;
    for (;;) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
        if ((++polls & 63u) == 0u) {
            if (t0 == 0) t0 = global_timer_ns();
            else if (global_timer_ns() - t0 > kBarrierTimeoutNs) return false;
        }
    }
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---- arithmetic --------------------------------------------------------------------------------------------------------
// Sum over the warp of values below 2^103 (all lanes get it): four 32-bit reductions.
__device__ __forceinline__ u128 warp_total_u128(u128 v)
{
    const unsigned m = 0x7ffffffu;
    const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)v & m);
    const unsigned b = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 27) & m);
    const unsigned c = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 54) & m);
    const unsigned d = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 81) & m);
    return (u128)((ull)a + ((ull)b << 27)) + ((u128)((ull)c + ((ull)d << 27)) << 54);
}
__device__ __forceinline__ ull warp_max_u64(ull v)
{
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
    return ((ull)hi << 32) | lo;
}
// Rounded benefit / cost as ordered bits (positive doubles compare like integers); 0 for no benefit.
__device__ __forceinline__ ull chip_key(u128 ben, double inv_cost)
{
    const ull hi = (ull)(ben >> 64);
    double b = __ull2double_rn((ull)ben);
    if (hi != 0) b += __ull2double_rn(hi) * 18446744073709551616.0;
    return (ull)__double_as_longlong(b * inv_cost);
}

// Slot ranges on the cycle are unrolled (slot k + K is slot k one iteration later): the physical slots of [a, b] are one run or,
// part by part, two.
template <bool kCyclic>
__device__ __forceinline__ bool phys_part(int part, int a, int b, int K, int *lo, int *hi)
{
    if (!kCyclic) { *lo = a; *hi = b; return part == 0; }
    const bool wraps = a < K && b >= K;
    if (part == 1) { *lo = 0; *hi = b - K; return wraps; }
    *lo = a >= K ? a - K : a; *hi = wraps ? K - 1 : b >= K ? b - K : b;
    return part == 0;
}
// Bits [lo, hi] of the 32 slots of word w
__device__ __forceinline__ unsigned word_mask(int w, int lo, int hi)
{
    if (hi < 32 * w || lo > 32 * w + 31) return 0u;
    unsigned m = 0xffffffffu;
    if (lo > 32 * w) m &= 0xffffffffu << (lo & 31);
    if (hi < 32 * w + 31) m &= 0xffffffffu >> (31 - (hi & 31));
    return m;
}

// One channel (a device and a direction): what is booked on it, slot by slot.
struct ChipChannel {
    unsigned *some, *full;      // bit per slot: something is booked; all of it is
    int64_t *part;              // booked time of a slot with `some` and not `full`
};
// A transfer window takes all of slots [lo, hi] (none if lo > hi) and `need` ns of slot e: the last slot of an eviction, the first
// of a prefetch.
struct ChipWindow {
    int lo, hi, e;
    int64_t need;
};
__device__ __forceinline__ ChipWindow transfer_window(int dir, const int64_t *start, int a, int ap, int bp, int b, int64_t t)
{
    ChipWindow w;
    w.lo = dir ? bp + 2 : a; w.hi = dir ? b : ap - 2; w.e = dir ? bp + 1 : ap - 1;
    w.need = dir ? start[bp + 2] - (start[b + 1] - t) : start[a] + t - start[ap - 1];
    return w;
}

// ---- the timeline in shared memory -------------------------------------------------------------------------------------
struct ChipTimeline {
    int64_t *ex;                // [K] pressure minus capacity, without the tile's offset
    int64_t *start;             // [K + 1] slot clock ([2K + 1] unrolled in cyclic mode)
    int64_t *off;               // [tiles of 32 slots] amount to add to every slot of the tile
    longlong2 *mm;              // [tiles] smallest and largest value with it
    int *stamp;                 // [tiles] iteration after which the tile changed last
};

__device__ __forceinline__ longlong2 tile_extremes_warp(const ChipTimeline &T, int K, int t, int lane)
{
    const int k = t * kTileO + lane;
    const bool in = k < K;
    const ull v = in ? (ull)(T.ex[k] + T.off[t]) ^ (1ull << 63) : 0ull;      // (signed order as unsigned order)
    const unsigned hi = (unsigned)(v >> 32), lo = (unsigned)v;
    const unsigned xh = __reduce_max_sync(0xffffffffu, in ? hi : 0u);
    const unsigned nh = __reduce_min_sync(0xffffffffu, in ? hi : 0xffffffffu);
    const unsigned xl = __reduce_max_sync(0xffffffffu, in && hi == xh ? lo : 0u);
    const unsigned nl = __reduce_min_sync(0xffffffffu, in && hi == nh ? lo : 0xffffffffu);
    longlong2 r;
    r.x = (long long)((((ull)nh << 32) | nl) ^ (1ull << 63));
    r.y = (long long)((((ull)xh << 32) | xl) ^ (1ull << 63));
    return r;
}

// Exact benefit of the (unrolled) absent range [a, b] for a tensor of s bytes, by one warp; every lane gets it.  A lane per tile: one
// at least s above capacity throughout counts s for all its time, one within capacity nothing; the few others are read slot by slot.
template <bool kCyclic>
__device__ __forceinline__ u128 benefit_warp(const ChipTimeline &T, int64_t s, int a, int b, int K, int lane)
{
    ull time = 0;
    u128 sum = 0;
#pragma unroll 1
    for (int part = 0; part < (kCyclic ? 2 : 1); ++part) {
        int lo, hi;
        if (!phys_part<kCyclic>(part, a, b, K, &lo, &hi)) break;
#pragma unroll 1
        for (int t0 = lo >> 5; t0 <= hi >> 5; t0 += 32) {
            const int t = t0 + lane;
            bool mixed = false;
            if (t <= hi >> 5) {
                const int k_lo = t * kTileO > lo ? t * kTileO : lo, k_hi = t * kTileO + kTileO - 1 < hi ? t * kTileO + kTileO - 1 : hi;
                const longlong2 mm = T.mm[t];
                const ull span = (ull)(T.start[k_hi + 1] - T.start[k_lo]);
                if (mm.x >= s) time += span;
                else mixed = mm.y > 0;
            }
            unsigned m = __ballot_sync(0xffffffffu, mixed);
#pragma unroll 1
            while (m) {
                const int tt = t0 + __ffs(m) - 1, k = tt * kTileO + lane;
                m &= m - 1;
                if (k >= lo && k <= hi) {
                    int64_t e = T.ex[k] + T.off[tt];
                    const ull dur = (ull)(T.start[k + 1] - T.start[k]);
                    e = e > s ? s : e < 0 ? 0 : e;
                    sum += (u128)(ull)e * (u128)dur;
                }
            }
        }
    }
    return warp_total_u128(sum + (u128)time * (u128)(ull)s);
}

// Of the lanes with `in`: the one with the exactly best candidate.
__device__ __noinline__ int contest(bool in, ull ben_hi, ull ben_lo, ull cost, int idx)
{
    Cand x, best;
    x.ben = ((u128)ben_hi << 64) | ben_lo; x.cost = cost; x.idx = in ? idx : -1; x.dest = 0;
    best.dest = 0;
    int f = 0;
    unsigned b = __ballot_sync(0xffffffffu, in);
#pragma unroll 1
    while (b) {
        f = __ffs(b) - 1;
        best.ben = ((u128)__shfl_sync(0xffffffffu, ben_hi, f) << 64) | __shfl_sync(0xffffffffu, ben_lo, f);
        best.cost = __shfl_sync(0xffffffffu, cost, f); best.idx = __shfl_sync(0xffffffffu, idx, f);
        b = __ballot_sync(0xffffffffu, (threadIdx.x & 31) != (unsigned)f && cand_beats(x, best));
    }
    return f;
}

// ---- a period's slot ranges --------------------------------------------------------------------------------------------
// A range [lo, hi] of slots is one word, (kSlotTop - lo) | hi << 16, so that two of them are compared with one subtraction:
// they meet iff hi1 - lo2 and hi2 - lo1 are both >= 0, and a guard bit above either half tells.
// (0 is the word of a range that meets none; the guard bits are free for flags)
constexpr unsigned kSlotTop = 0x7fff, kGuard = 0x80008000u;
__device__ __forceinline__ unsigned range_word(int lo, int hi) { return (kSlotTop - (unsigned)lo) | (unsigned)hi << 16; }
__device__ __forceinline__ int range_lo(unsigned w) { return (int)(kSlotTop - (w & kSlotTop)); }
__device__ __forceinline__ int range_hi(unsigned w) { return (int)(w >> 16); }
// The same range seen from the other side; the ranges of the winner are brought into this form once.
__device__ __forceinline__ unsigned probe_word(int lo, int hi) { return (kSlotTop - (unsigned)hi) | (unsigned)lo << 16; }
// On the cycle a range also meets one that lies an iteration earlier or later.
template <bool kCyclic>
struct ChipProbe {
    unsigned p[kCyclic ? 3 : 1];
    __device__ __forceinline__ ChipProbe(int lo, int hi, int K)
    {
        p[0] = probe_word(lo, hi);
        if (kCyclic) {
            const unsigned never = probe_word(0, 0) | (unsigned)kSlotTop << 16;
            p[kCyclic ? 1 : 0] = lo + K >= (int)kSlotTop ? never : probe_word(lo + K, hi + K >= (int)kSlotTop ? (int)kSlotTop - 1 : hi + K);
            p[kCyclic ? 2 : 0] = hi - K < 0 ? never : probe_word(lo - K < 0 ? 0 : lo - K, hi - K);
        }
    }
    // 0 if they meet
    __device__ __forceinline__ unsigned misses(unsigned w) const
    {
        unsigned m = ~((w | kGuard) - p[0]) & kGuard;
        if (kCyclic) {
            const unsigned a = ~((w | kGuard) - p[kCyclic ? 1 : 0]) & kGuard, b = ~((w | kGuard) - p[kCyclic ? 2 : 0]) & kGuard;
            m = m < a ? m : a;
            m = m < b ? m : b;
        }
        return m;
    }
};

// A period's data: size (40 bits), transfer time to the current destination and to the host (44 bits each: usable destinations
// only).
__device__ __forceinline__ ulonglong2 pack_data(int64_t s, int64_t t, ull th)
{
    ulonglong2 d;
    d.x = (ull)s | (ull)t << 40;
    d.y = (ull)t >> 24 | th << 20;
    return d;
}
__device__ __forceinline__ int64_t data_size(ulonglong2 d) { return (int64_t)(d.x & 0xffffffffffull); }
__device__ __forceinline__ int64_t data_time(ulonglong2 d) { return (int64_t)(d.x >> 40 | (d.y & 0xfffffull) << 24); }
__device__ __forceinline__ ull data_rest(ulonglong2 d) { return d.y >> 20; }

// The periods of a block are looked at in at most 32 groups (one per lane of the warp that looks for the best) of 32, 64 or 128.
__host__ __device__ inline int chip_group_log(int64_t per_block) { return per_block <= 1024 ? 0 : per_block <= 2048 ? 1 : 2; }
__host__ __device__ inline int64_t chip_padded(int64_t per_block)
{
    const int64_t g = (int64_t)32 << chip_group_log(per_block);
    return (per_block + g - 1) / g * g;
}
__host__ __device__ inline size_t chip_round(size_t x) { return (x + 15) / 16 * 16; }
// Shared memory for candidates, timeline and periods ...
__host__ __device__ inline size_t chip_smem_core(int64_t K, int64_t per_block, int C, bool host_cap, bool cyclic)
{
    const size_t nt = (size_t)((K + kTileO - 1) / kTileO), np = (size_t)chip_padded(per_block);
    return (size_t)2 * C * sizeof(ChipCand) + chip_round((size_t)K * 8) + chip_round((size_t)((cyclic ? 2 * K : K) + 1) * 8) +
           chip_round(nt * 8) + nt * 16 + 9 * chip_round(nt * 4) + (host_cap ? chip_round(nt * 8) : 0) + np * (8 + 16 + 8 + 8 + 8 + 4 * 4);
}
// ... and for the booked amounts.
__host__ __device__ inline size_t chip_smem_busy(int64_t K, bool host_cap) { return chip_round((size_t)K * 8) * (host_cap ? 5 : 4); }

template <bool kBatch, bool kCyclic>
__global__ void __launch_bounds__(kChipThreads, 1) k_plan_chip(PlanArgs A, ChipArgs O, BatchArgs B)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ ull s_bar[2];
    __shared__ ChipWinner s_win;
    __shared__ ull s_gkey[32];                          // of each group of periods: the best, and its key
    __shared__ int s_gtop[32];
    __shared__ int64_t s_moved[2];                      // bytes sent to the SSD and to host memory
    __shared__ ull s_floor;                             // best exact key known in this iteration
    __shared__ int s_over;                              // tiles above capacity
    __shared__ unsigned s_bits;
    __shared__ long long s_pk[kChipWarps];
    __shared__ int s_ps[kChipWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int K = (int)A.K;
    const int64_t Pn64 = *A.Pn_dev < A.geo_stride ? *A.Pn_dev : A.geo_stride;
    const int64_t *P_src = A.P;
    uint64_t bw0 = A.bw[G10_DEST_SSD], bw1 = A.bw[G10_DEST_HOST];
    const int64_t *var_dur = nullptr;
    if (kBatch) {
        const int v = blockIdx.x / C;
        const BatchVariant var = B.variants[v];
        A.fits_always = var.cap >= ((uint64_t)1 << 63) ? 1 : 0;
        A.cap = A.fits_always ? INT64_MAX : (int64_t)var.cap;
        A.host_capacity = var.host_capacity;
        A.out += (size_t)v * A.out_cap;
        A.summary += (size_t)v * 8;
        P_src = B.P0;
        A.P = B.P_out + (size_t)v * K;
        bw0 = var.ssd_bw; bw1 = var.host_bw;
        var_dur = var.kernel_ns;
    }
    const bool host_cap = A.host_capacity != 0;
    unsigned dev_bits = 0;                              // device status bits of this plan
    const int64_t per_block = (Pn64 + C - 1) / C;
    // Does it fit?  (The answer is the same in all blocks, and in all variants of a batch: the host asks variant 0.)
    const bool host_room = kBatch ? B.host_cap != 0 : host_cap;
    bool fits = (kCyclic ? 2 * A.K : A.K) < (int64_t)kSlotTop && per_block <= kChipMaxPeriods, busy_smem = false;
    if (fits) {
        const size_t core = chip_smem_core(A.K, per_block, C, host_room, kCyclic);
        busy_smem = core + chip_smem_busy(A.K, host_room) <= (size_t)O.smem_bytes;
        fits = core <= (size_t)O.smem_bytes && (busy_smem || (O.busy_global && A.K <= kChipMaxSlots));
    }
    if (!fits) {
        if ((kBatch || kCyclic) && tid == 0 && rank == 0) {
            for (int j = 0; j < 7; ++j) A.summary[j] = j == 2 || j == 4 ? -1 : 0;
            A.summary[7] = G10_DEV_BATCH_UNFIT;
        }
        return;
    }
    const int Pn = (int)Pn64, np = (int)chip_padded(per_block), lq = chip_group_log(per_block), NG = np >> (5 + lq);
    const int nl = Pn > rank ? (Pn - rank + C - 1) / C : 0;        // this block's periods: rank, rank + C, ...
    const int64_t limit = (A.max_iterations <= 0 || A.max_iterations > Pn64) ? Pn64 : A.max_iterations;
    const int NT = (K + kTileO - 1) / kTileO;
    // group g belongs to warp g mod kChipWarps; the j-th period of this lane
    const int mine = NG > warp ? ((NG - warp + kChipWarps - 1) / kChipWarps) << lq : 0;
    auto entry = [&](int j) { return ((((j >> lq) * kChipWarps + warp) << lq) + (j & ((1 << lq) - 1))) * 32 + lane; };

    unsigned char *at = smem_raw;
    auto take = [&](size_t bytes) { unsigned char *p = at; at += chip_round(bytes); return p; };
    ChipCand *s_block = (ChipCand *)take((size_t)2 * C * sizeof(ChipCand));  // the best period of every block, two exchanges in turn
    ChipTimeline T;
    T.ex = (int64_t *)take((size_t)K * 8);
    T.start = (int64_t *)take((size_t)((kCyclic ? 2 * K : K) + 1) * 8);
    T.off = (int64_t *)take((size_t)NT * 8); T.mm = (longlong2 *)take((size_t)NT * 16);
    T.stamp = (int *)take((size_t)NT * 4);
    const unsigned bit_words = (unsigned)chip_round((size_t)NT * 4) / 4;
    unsigned *bits = (unsigned *)take((size_t)8 * bit_words * 4);  // some / full of SSD out, SSD in, host out, host in
    int64_t *hmax = (int64_t *)(host_cap ? take((size_t)NT * 8) : nullptr);     // largest host occupancy per tile
    // the periods: slots of the eviction window (bit 15: destination) and of the prefetch window, data, rounded score (0: none,
    // erased), inverse of the cost, benefit, absent slots (current destination; host), iteration in which it was scored last
    uint2 *cwin = (uint2 *)take((size_t)np * 8);
    ulonglong2 *cdata = (ulonglong2 *)take((size_t)np * 16);
    ull *ckey = (ull *)take((size_t)np * 8);
    double *cinv = (double *)take((size_t)np * 8);
    ull *cben = (ull *)take((size_t)np * 8);
    unsigned *cben_hi = (unsigned *)take((size_t)np * 4), *cabs = (unsigned *)take((size_t)np * 4), *chost = (unsigned *)take((size_t)np * 4);
    int *cstamp = (int *)take((size_t)np * 4);
    int64_t *busy = busy_smem ? (int64_t *)take((size_t)K * 8 * 4) : O.busy_global + (size_t)rank * 4 * K;
    int64_t *hocc = !host_cap ? nullptr : busy_smem ? (int64_t *)take((size_t)K * 8) : O.hocc_global + (size_t)rank * K;
    auto channel = [&](int X, int dir) {
        ChipChannel c;
        const unsigned j = (unsigned)(2 * X + dir);
        c.some = bits + j * 2u * bit_words;
        c.full = c.some + bit_words;
        c.part = busy + (size_t)j * K;
        return c;
    };
    // (re)starts period li with absent slots r on destination X: its first bound is the benefit it would have if the whole range
    // were at least s above capacity
    auto begin_period = [&](int li, int X, int a, int b, unsigned r, int64_t s, int64_t t, ull th) {
        const int ap = range_lo(r), bp = range_hi(r);
        const ull span = (ull)(T.start[bp + 1] - T.start[ap]);
        const u128 ben = (u128)(ull)s * (u128)span;
        const double inv = 1.0 / __ull2double_rn(2ull * (ull)t);
        cdata[li] = pack_data(s, t, th);
        cinv[li] = inv; cben[li] = (ull)ben; cben_hi[li] = (unsigned)(ben >> 64); ckey[li] = chip_key(ben, inv);
        cwin[li] = make_uint2(range_word(a, ap - 1) | (unsigned)X << 15, range_word(bp + 1, b));
        cabs[li] = r; cstamp[li] = -1;
    };
    // the best of a group of periods (one warp)
    auto update_group = [&](int g) {
        const int first = (g << (5 + lq)) + lane;
        ull k = ckey[first];
        int li = first;
        if (lq > 0) {
#pragma unroll 1
            for (int n = 1; n < 1 << lq; ++n) {
                const int ln = first + n * 32;
                const ull kn = ckey[ln];
                bool take = kn > k;
                if (k != 0 && kn + kBand >= k && k + kBand >= kn) {
                    Cand x, y;                                // too close to call by the rounded scores: by the exact ones
                    x.ben = ((u128)cben_hi[ln] << 64) | cben[ln]; x.cost = 2ull * (ull)data_time(cdata[ln]); x.idx = ln;
                    y.ben = ((u128)cben_hi[li] << 64) | cben[li]; y.cost = 2ull * (ull)data_time(cdata[li]); y.idx = li;
                    take = cand_beats(x, y);
                }
                if (take) { k = kn; li = ln; }
            }
        }
        const ull m = warp_max_u64(k);
        const bool in = k + kBand >= m && k != 0;
        const unsigned b = __ballot_sync(0xffffffffu, in);
        int l = b ? __ffs(b) - 1 : 0;
        if (b & (b - 1u)) l = contest(in, (ull)cben_hi[li], cben[li], 2ull * (ull)data_time(cdata[li]), li);
        if (lane == l) { s_gkey[g] = k; s_gtop[g] = li; }
        __syncwarp();
    };

    // ---------------- the timeline and the periods
    if (tid == 0) {
        s_over = 0; s_bits = 0; s_moved[0] = s_moved[1] = 0;
        bar_init(smem_addr(&s_bar[0]), 1); bar_init(smem_addr(&s_bar[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
#pragma unroll 1
    for (int k = tid; k < K; k += kChipThreads) T.ex[k] = P_src[k] - A.cap;
    if (!kBatch) {
#pragma unroll 1
        for (int k = tid; k <= (kCyclic ? 2 * K : K); k += kChipThreads) T.start[k] = A.start[k];
    } else {
        // slot clock of this variant: exclusive scan of its durations (each thread a run of consecutive kernels);
        // a duration outside [1, 2^44) counts as 1 and raises the status bit, as in the trace-level pass
        const int chunk = (K + kChipThreads - 1) / kChipThreads;
        const int k0 = tid * chunk < K ? tid * chunk : K, k1 = k0 + chunk < K ? k0 + chunk : K;
        long long sum = 0;
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            long long d = var_dur[k];
            if (d < 1 || d >= ((long long)1 << 44)) { d = 1; dev_bits |= G10_DEV_BAD_DURATION; }
            sum += d;
        }
        const long long incl = warp_inclusive_scan_i64(sum, lane);
        if (lane == 31) s_pk[warp] = incl;
        __syncthreads();
        long long run = incl - sum;
#pragma unroll 1
        for (int w = 0; w < warp; ++w) run += s_pk[w];
#pragma unroll 1
        for (int k = k0; k < k1; ++k) {
            long long d = var_dur[k];
            if (d < 1 || d >= ((long long)1 << 44)) d = 1;
            T.start[k] = run;
            run += d;
        }
        if (k1 == K) T.start[K] = run;                 // every thread at or past the end holds the total
    }
#pragma unroll 1
    for (int t = tid; t < NT; t += kChipThreads) {
        T.off[t] = 0; T.stamp[t] = 0;
        if (host_cap) hmax[t] = 0;
    }
#pragma unroll 1
    for (int j = tid; j < 8 * (int)bit_words; j += kChipThreads) bits[j] = 0;
    if (host_cap)
#pragma unroll 1
        for (int k = tid; k < K; k += kChipThreads) hocc[k] = 0;
    __syncthreads();                                   // (the clock is complete)
    if (kBatch && T.start[K] >= ((int64_t)1 << 44)) {
        // (transfer times of the periods have to fit 44 bits; a trace's own clock is checked where it is made)
        if (tid == 0 && rank == 0) {
            for (int j = 0; j < 7; ++j) A.summary[j] = j == 2 || j == 4 ? -1 : 0;
            A.summary[7] = G10_DEV_BAD_DURATION;
        }
        return;
    }
#pragma unroll 1
    for (int li = tid; li < np; li += kChipThreads) {
        ckey[li] = 0; cwin[li] = make_uint2(0, 0); chost[li] = kNoRange;
        if (li >= nl) continue;
        const int p = li * C + rank;
        const int u = A.per_u[p], v = A.per_v[p];
        const int64_t s = A.bytes[A.per_t[p]];
        // nothing is booked yet: the first usable destination it is, SSD before host
        int dest = -1;
        unsigned r = kNoRange;
        int64_t t = 0, th = 0;
#pragma unroll 1
        for (int X = 1; X >= 0; --X) {
            int ap, bp;
            int64_t tx;
            if (kBatch || O.alone) period_geometry(T.start, u, v, s, X ? bw1 : bw0, &tx, &ap, &bp);
            else { ap = A.geo_a[X * A.geo_stride + p]; bp = A.geo_b[X * A.geo_stride + p]; tx = A.geo_t[X * A.geo_stride + p]; }
            if (X == G10_DEST_HOST && host_cap && (uint64_t)s > A.host_capacity) ap = -1;            // (never fits there)
            if (ap < 0) continue;
            dest = X; t = tx;
            r = range_word(ap, bp);
            if (X == G10_DEST_HOST) { th = tx; chost[li] = r; }
        }
        if (dest >= 0) begin_period(li, dest, u + 1, v - 1, r, s, t, (ull)th);
    }
#pragma unroll 1
    for (int t = warp; t < NT; t += kChipWarps) {
        const longlong2 mm = tile_extremes_warp(T, K, t, lane);
        if (lane == 0) { T.mm[t] = mm; if (mm.y > 0) atomicAdd(&s_over, 1); }
    }
    __syncthreads();

    unsigned groups = 0xffffffffu;                     // groups of this warp (bit i: its i-th) whose best has to be found again
    int64_t n_mig = 0, rounds = 0;
    int status = -1;
    // A little less than the last winner's key.  Warp 0's alone: in the others it stays 0, and with it `least` below.  They have to
    // rescore whatever may win when they are asked for help: warp 0 lowers its own `least` when a bound turns out in front, and
    // helpers that kept a higher one would leave everything to it (a variant of this search, three ViT-H steps at half their peak:
    // 25.6 ms with such helpers, 15.7 without).
    ull likely = 0;
    unsigned sent = 0;                                 // exchanges with the other blocks so far
#pragma unroll 1
    for (int64_t it64 = 0;; ++it64) {
#pragma unroll 1
        for (int g = warp; g < NG; g += kChipWarps, groups >>= 1) if (groups & 1u) update_group(g);
        if (it64 == 0 && C > 1) cluster_sync_all();    // (the transaction barriers are set up everywhere)
        else __syncthreads();
        if (A.fits_always || s_over == 0) { status = n_mig == 0 ? G10_ALREADY_FITS : G10_FIT; break; }
        if (it64 >= limit) { status = limit < Pn64 ? G10_ITERATION_LIMIT : G10_EXHAUSTED; break; }
        rounds += 1;
        const int it = (int)it64;
        // ---------------- S: the winner.  Warp 0 takes the best period by bound; if its score is not exact any more it rescores it
        // and looks again.  After a few of those it asks the other warps for help: each rescores the best of its own groups, as
        // long as they may beat the best exact score.
        ull floor = 0;
        bool help = false, fresh = true;
        ull least = C > 1 ? likely : 0ull;                    // bounds below this are not made exact unless it turns out necessary
#pragma unroll 1
        for (;;) {
            int top = -1;
            if (warp == 0 || help) {
                int done = 0;
#pragma unroll 1
                for (;;) {
                    ull k = lane < NG ? s_gkey[lane] : 0ull;
                    if (help && (lane & (kChipWarps - 1)) != warp) k = 0;
                    const ull m = warp_max_u64(k);
                    top = -1;
                    fresh = true;
                    if (m == 0 || (help && m + kBand < s_floor)) break;
                    const bool in = k + kBand >= m && k != 0;
                    const unsigned b = __ballot_sync(0xffffffffu, in);
                    int l = __ffs(b) - 1;
                    if ((b & (b - 1u)) != 0u && !help) {
                        const int q = in ? s_gtop[lane] : 0;
                        l = contest(in, (ull)cben_hi[q], cben[q], 2ull * (ull)data_time(cdata[q]), q);
                    }
                    top = s_gtop[l];
                    if (m < least) { fresh = false; break; }  // (far from winning, in all likelihood: it goes out as a bound)
                    // Is its score exact?  It is if no tile of its absent range has changed since it was found (never, for the first
                    // bound) -- or if the tile is still at least the tensor's size above capacity throughout, so that it was before
                    // and counts the same.
                    const int stamp = cstamp[top];
                    const unsigned r = cabs[top];
                    const int64_t s = data_size(cdata[top]);
                    const int ra = range_lo(r), rb = range_hi(r);
                    bool hit = false;
                    if (stamp != it)
#pragma unroll 1
                        for (int part = 0; part < (kCyclic ? 2 : 1); ++part) {
                            int lo, hi;
                            if (!phys_part<kCyclic>(part, ra, rb, K, &lo, &hi)) break;
#pragma unroll 1
                            for (int t = (lo >> 5) + lane; t <= hi >> 5; t += 32) hit |= T.stamp[t] > stamp && T.mm[t].x < s;
                        }
                    if (!__any_sync(0xffffffffu, hit)) break;
                    if (done == kAlone) { top = -2; break; }
                    ++done;
                    const u128 ben = benefit_warp<kCyclic>(T, s, ra, rb, K, lane);
                    const ull key = chip_key(ben, cinv[top]);
                    if (key > floor) floor = key;
                    if (lane == 0) { cben[top] = (ull)ben; cben_hi[top] = (unsigned)(ben >> 64); ckey[top] = key; cstamp[top] = it; }
                    __syncwarp();
                    update_group(top >> (5 + lq));
                }
            }
            if (warp == 0 && !help) {
                if (lane == 0) s_floor = floor;
                int what = top == -2 ? kHelp : top < 0 ? kNone : kFound;
                if (top != -2) {
                    const int li = top < 0 ? 0 : top;
                    const uint2 win = cwin[li];
                    ChipCand w;
                    w.key = top < 0 ? 0ull : ckey[li]; w.ben_lo = cben[li]; w.data = cdata[li];
                    w.rec = make_uint4(win.x, win.y, cabs[li], cben_hi[li]);
                    int idx = top * C + rank;
                    if (C > 1) {
                        // to all blocks of the cluster, and the best of theirs (the period goes where the transfer time to the
                        // host was; the top bit of the first range says that the key is exact)
                        ChipCand *from = s_block + (sent & 1u) * C;
                        const unsigned bar = smem_addr(&s_bar[sent & 1u]);
                        if (lane == 0) bar_expect(bar, (unsigned)(C * sizeof(ChipCand)));
                        w.data.y = (w.data.y & 0xfffffull) | (ull)(unsigned)idx << 20;
                        w.rec.x = (w.rec.x & 0x7fffffffu) | (fresh ? 0x80000000u : 0u);
                        const unsigned part = (unsigned)lane % 3u;
                        uint4 v = w.rec;
                        if (part == 0) v = make_uint4((unsigned)w.key, (unsigned)(w.key >> 32), (unsigned)w.ben_lo, (unsigned)(w.ben_lo >> 32));
                        if (part == 1) v = make_uint4((unsigned)w.data.x, (unsigned)(w.data.x >> 32), (unsigned)w.data.y, (unsigned)(w.data.y >> 32));
#pragma unroll 1
                        for (int j = lane; j < 3 * C && lane < 30; j += 30)
                            st_async_v4(peer_addr(smem_addr(&from[rank]) + 16 * part, (unsigned)(j / 3)), v, peer_addr(bar, (unsigned)(j / 3)));
                        const bool here = bar_wait(bar, sent >> 1 & 1u);
                        sent += 1;
                        if (!__all_sync(0xffffffffu, here)) what = kGaveUp;
                        else {
                            const ChipCand y = from[lane < C ? lane : 0];
                            const ull k = lane < C ? y.key : 0ull, m = warp_max_u64(k);
                            const bool in = k + kBand >= m && k != 0, exact = (y.rec.x >> 31) != 0u;
                            const unsigned b = __ballot_sync(0xffffffffu, in);
                            what = m == 0 ? kNone : kFound;
                            int l = b ? __ffs(b) - 1 : 0;
                            if (__any_sync(0xffffffffu, in && !exact)) {
                                // a bound is in front: the blocks whose bound may beat the best exact key make it exact
                                least = warp_max_u64(exact ? k : 0ull);
                                least = least > kBand ? least - kBand : 1ull;
                                continue;
                            }
                            if (b & (b - 1u)) l = contest(in, (ull)y.rec.w, y.ben_lo, 2ull * (ull)data_time(y.data), (int)data_rest(y.data));
                            w = from[l];
                            idx = (int)data_rest(w.data);
                            w.rec.x &= 0x7fffffffu;
                            likely = (ull)__double_as_longlong(__longlong_as_double((long long)w.key) * 0.97);
                        }
                    }
                    if (lane == 0) { s_win.c = w; s_win.idx = idx; }
                }
                if (lane == 0) s_win.what = what;
            }
            __syncthreads();
            if (help) help = false;
            else if (s_win.what != kHelp) break;
            else { help = true; floor = s_floor; }
        }
        // ---------------- C: the winner is applied
        const int what = s_win.what;
        if (what == kGaveUp) { status = -2; break; }
        if (what == kNone) { status = G10_EXHAUSTED; break; }
        const uint4 wr = s_win.c.rec;
        const int wa = range_lo(wr.x), wap = range_lo(wr.z), wbp = range_hi(wr.z), wb = range_hi(wr.y), X = (int)(wr.x >> 15 & 1u);
        const ChipProbe<kCyclic> p_out(wa, wap - 1, K), p_in(wbp + 1, wb, K);
        const ulonglong2 wd = s_win.c.data;
        const int64_t ws = data_size(wd);
        // pressure falls by its size in the absent slots: whole tiles by their offset, the tiles at the ends slot by slot
#pragma unroll 1
        for (int part = 0; part < (kCyclic ? 2 : 1); ++part) {
            int lo, hi;
            if (!phys_part<kCyclic>(part, wap, wbp, K, &lo, &hi)) break;
            if (part) __syncthreads();                        // (the two parts may share a tile)
            const int ta = lo >> 5, tb = hi >> 5, fa = (lo + 31) >> 5, fb = ((hi + 1) >> 5) - 1;
#pragma unroll 1
            for (int t = fa + tid; t <= fb; t += kChipThreads) {
                longlong2 mm = T.mm[t];
                const bool was = mm.y > 0;                    // (a tile within capacity counts nothing, before and after)
                mm.x -= ws; mm.y -= ws;
                T.off[t] -= ws; T.mm[t] = mm;
                if (was) { T.stamp[t] = it + 1; if (mm.y <= 0) atomicSub(&s_over, 1); }
            }
            int t = -1;
            if (warp == kChipWarps - 1 && ta < fa) t = ta;
            if (warp == kChipWarps - 2 && tb > fb && !(tb == ta && ta < fa)) t = tb;
            if (t >= 0) {
                const int k = t * kTileO + lane;
                if (k >= lo && k <= hi) T.ex[k] -= ws;
                const longlong2 mm = tile_extremes_warp(T, K, t, lane);
                if (lane == 0) {
                    if (T.mm[t].y > 0) { T.stamp[t] = it + 1; if (mm.y <= 0) atomicSub(&s_over, 1); }
                    T.mm[t] = mm;
                }
            }
        }
        // its transfer windows are booked (a warp each)
        if (warp == kChipWarps - 3 || warp == kChipWarps - 4) {
            const int dir = kChipWarps - 3 - warp;
            const ChipChannel c = channel(X, dir);
            const ChipWindow w = transfer_window(dir, T.start, wa, wap, wbp, wb, data_time(wd));
            const int slo = w.lo <= w.hi && w.lo < w.e ? w.lo : w.e, shi = w.lo <= w.hi && w.hi > w.e ? w.hi : w.e;
#pragma unroll 1
            for (int part = 0; part < (kCyclic ? 2 : 1); ++part) {
                int lo, hi;
                if (!phys_part<kCyclic>(part, slo, shi, K, &lo, &hi)) break;
                const int shift = kCyclic && (part || slo >= K) ? K : 0, e = w.e - shift;
                __syncwarp();
#pragma unroll 1
                for (int i = (lo >> 5) + lane; i <= hi >> 5; i += 32) {
                    const unsigned old = c.some[i], m = word_mask(i, lo, hi);
                    if (e >= lo && e <= hi && e >> 5 == i) c.part[e] = (old >> (e & 31) & 1u ? c.part[e] : 0) + w.need;
                    c.some[i] = old | m;
                    if (w.lo <= w.hi) c.full[i] |= m & word_mask(i, w.lo - shift, w.hi - shift);
                }
            }
        }
        if (X == G10_DEST_HOST && host_cap)
#pragma unroll 1
            for (int part = 0; part < (kCyclic ? 2 : 1); ++part) {
                int lo, hi;
                if (!phys_part<kCyclic>(part, wa, wb, K, &lo, &hi)) break;
                if (part) __syncthreads();
#pragma unroll 1
                for (int t = (lo >> 5) + warp; t <= hi >> 5; t += kChipWarps) {
                    const int k = t * kTileO + lane;
                    int64_t h = 0;
                    if (k < K) {
                        h = hocc[k];
                        if (k >= lo && k <= hi) hocc[k] = h += ws;
                    }
                    const ull m = warp_max_u64((ull)h);
                    if (lane == 0) hmax[t] = (int64_t)m;
                }
            }
        if (tid == kChipThreads - 5 * 32) {                   // (one thread keeps the account)
            const int64_t t = data_time(wd);
            if (rank == 0 && n_mig < A.out_cap) {
                g10_migration m;
                m.period = s_win.idx; m.tensor = 0; m.dest = X; m.absent_first = wap; m.absent_last = wbp; m.iteration = it;
                m.evict_issue_ns = T.start[wa]; m.prefetch_issue_ns = T.start[wb + 1] - t; m.transfer_ns = t;
                A.out[n_mig] = m;
            } else if (rank == 0) dev_bits |= G10_DEV_PLAN_OVERFLOW;
            s_moved[X] += ws;
        }
        n_mig += 1;
        // which of this lane's periods have a window on the channels that have just been booked?
        unsigned check = 0;                                   // (bit j: its j-th)
        {
            const bool all_host = X == G10_DEST_HOST && host_cap;
            const unsigned flag = (unsigned)X << 15;
#pragma unroll 2
            for (int j = 0; j < mine; ++j) {
                const uint2 q = cwin[entry(j)];
                const unsigned mo = p_out.misses(q.x), mi = p_in.misses(q.y);
                unsigned miss = mo < mi ? mo : mi;
                if (all_host && q.y != 0u) miss = 0u;
                if ((miss | ((q.x ^ flag) & 0x8000u)) == 0u) check |= 1u << j;
            }
        }
        groups = 0;
        if (!__syncthreads_or(check != 0u)) continue;
        // ---------------- those periods (the winner is among them, in its block): is their destination still possible?  Not if a
        // slot that a window needs wholly has been booked, or if the slot it needs in part has too little left.  Then the host, if
        // its windows are free.
        const int widx = s_win.idx;
#pragma unroll 1
        while (check) {
            const int j = __ffs(check) - 1, li = entry(j);
            check &= check - 1;
            const uint2 q = cwin[li];
            const ulonglong2 d = cdata[li];
            const int a = range_lo(q.x), b = range_hi(q.y);
            const int64_t s = data_size(d);
            unsigned r = cabs[li];
            int64_t t = data_time(d);
            int D = X;
            bool free = li * C + rank != widx;
#pragma unroll 1
            for (;;) {
#pragma unroll 1
                for (int dir = 0; dir < 2 && free; ++dir) {
                    const ChipWindow w = transfer_window(dir, T.start, a, range_lo(r), range_hi(r), b, t);
                    const ChipProbe<kCyclic> &p = dir ? p_in : p_out;
                    const bool again = D != X;                // (a new destination: the whole window has to be looked at)
                    if (!again && w.lo <= w.hi && p.misses(range_word(w.lo, w.hi)) == 0u) { free = false; break; }
                    if (!again && p.misses(range_word(w.e, w.e)) != 0u) continue;
                    const ChipChannel c = channel(D, dir);
                    const int e = kCyclic && w.e >= K ? w.e - K : w.e;
                    const unsigned some = c.some[e >> 5] >> (e & 31) & 1u, full = c.full[e >> 5] >> (e & 31) & 1u;
                    if (some && (full || c.part[e] + w.need > T.start[w.e + 1] - T.start[w.e])) { free = false; break; }
                    if (!again || w.lo > w.hi) continue;
                    unsigned any = 0;
#pragma unroll 1
                    for (int part = 0; part < (kCyclic ? 2 : 1); ++part) {
                        int lo, hi;
                        if (!phys_part<kCyclic>(part, w.lo, w.hi, K, &lo, &hi)) break;
#pragma unroll 2
                        for (int i = lo >> 5; i <= hi >> 5; ++i) any |= c.some[i] & word_mask(i, lo, hi);
                    }
                    free = any == 0u;
                }
                if (free && D == G10_DEST_HOST && host_cap) {
                    const int64_t most = (int64_t)(A.host_capacity > (uint64_t)INT64_MAX ? (uint64_t)INT64_MAX : A.host_capacity) - s;
#pragma unroll 1
                    for (int part = 0; part < (kCyclic ? 2 : 1); ++part) {
                        int lo, hi;
                        if (!phys_part<kCyclic>(part, a, b, K, &lo, &hi)) break;
#pragma unroll 1
                        for (int k = lo; k <= hi && free; ) {
                            const int end = (k | 31) < hi ? k | 31 : hi;
                            if (hmax[k >> 5] <= most) { k = end + 1; continue; }
                            for (; k <= end; ++k) if (hocc[k] > most) free = false;
                        }
                    }
                }
                if (free || D == G10_DEST_HOST || chost[li] == kNoRange || li * C + rank == widx) break;
                r = chost[li];
                D = G10_DEST_HOST; t = (int64_t)data_rest(d); free = true;
            }
            if (free && D == X) continue;
            groups |= 1u << (j >> lq);
            if (free) begin_period(li, D, a, b, r, s, t, (ull)t);
            else { cwin[li] = make_uint2(0, 0); ckey[li] = 0; }
        }
        groups = __reduce_or_sync(0xffffffffu, groups);
    }
    // ---------------- epilogue: final pressure, peak and its lowest slot, summary
    dev_bits = __reduce_or_sync(0xffffffffu, dev_bits);
    if (lane == 0 && dev_bits) atomicOr(&s_bits, dev_bits);
    __syncthreads();
    if (C > 1) cluster_sync_all();                     // (nobody leaves while something may still be on its way to it)
    if (rank != 0) return;
    long long pk = 0;
    int ps = -1;
#pragma unroll 1
    for (int k = tid; k < K; k += kChipThreads) {
        const long long pv = T.ex[k] + T.off[k / kTileO] + A.cap;
        A.P[k] = pv;
        if (ps < 0 || pv > pk) { pk = pv; ps = k; }      // k ascending per thread: first maximum kept
    }
    // (the records' tensors, left out in the loop because they have to be looked up)
#pragma unroll 1
    for (int64_t j = tid; j < n_mig && j < A.out_cap; j += kChipThreads) A.out[j].tensor = A.per_t[A.out[j].period];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long yk = __shfl_xor_sync(0xffffffffu, pk, o);
        const int ys = __shfl_xor_sync(0xffffffffu, ps, o);
        if (ys >= 0 && (ps < 0 || yk > pk || (yk == pk && ys < ps))) { pk = yk; ps = ys; }
    }
    if (lane == 0) { s_pk[warp] = pk; s_ps[warp] = ps; }
    __syncthreads();
    if (tid == 0) {
#pragma unroll 1
        for (int j = 1; j < kChipWarps; ++j)
            if (s_ps[j] >= 0 && (ps < 0 || s_pk[j] > pk || (s_pk[j] == pk && s_ps[j] < ps))) { pk = s_pk[j]; ps = s_ps[j]; }
        if (status == -2) { raise_status(A.status, G10_DEV_TIMEOUT); s_bits |= G10_DEV_TIMEOUT; }
        A.summary[0] = n_mig; A.summary[1] = rounds; A.summary[2] = status == -2 ? -1 : status;
        A.summary[3] = ps < 0 ? 0 : pk; A.summary[4] = ps;
        A.summary[5] = s_moved[0]; A.summary[6] = s_moved[1];
        // status bits found by this plan: the batch keeps them per variant, a single plan in the call's status word
        if (O.alone) A.summary[7] = (int64_t)(s_bits | (unsigned)*(volatile ull *)A.status);
        else if (kBatch || kCyclic) A.summary[7] = s_bits;   // (the call-wide status word is folded in afterwards)
        else if (s_bits) raise_status(A.status, s_bits);
        if (!kBatch) *O.done = 1u;
    }
}

enum { kOnePlan, kOneCycle, kManyPlans };
static const void *chip_kernel(int which)
{
    return which == kOnePlan ? (const void *)k_plan_chip<false, false> : which == kOneCycle ? (const void *)k_plan_chip<false, true> : (const void *)k_plan_chip<true, false>;
}

// Shared memory a launch can offer (0 if a query fails).
static int chip_smem_budget(int which)
{
    static int known[3][kMaxDevices];
    return dynamic_smem_room(chip_kernel(which), known[which]);
}

// Blocks of the largest cluster that can be placed with that memory.
static int chip_largest(int which)
{
    static int known[3][kMaxDevices];
    const int room = chip_smem_budget(which);
    const void *kernel = chip_kernel(which);
    return room > 0 ? largest_cluster(&kernel, false, kChipThreads, (size_t)room, known[which]) : 0;
}

// Launches `plans` clusters of C blocks (one per plan).
static cudaError_t launch_chip(int which, PlanArgs A, ChipArgs O, BatchArgs B, int plans, int C, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(plans * C)); cfg.blockDim = dim3(kChipThreads); cfg.dynamicSmemBytes = (size_t)O.smem_bytes; cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    void *args[] = {&A, &O, &B};
    if (const cudaError_t e = allow_launch(chip_kernel(which), (size_t)O.smem_bytes, C); e != cudaSuccess) return e;
    return cudaLaunchKernelExC(&cfg, chip_kernel(which), args);
}

static ChipArgs chip_args(int which, const Workspace &w)
{
    ChipArgs O;
    O.done = w.one_done; O.smem_bytes = chip_smem_budget(which);
    O.busy_global = w.busy_rep; O.hocc_global = w.hocc_rep;
    O.alone = 0;
    return O;
}

// Blocks of the cluster.  Measured (ms): 96-kernel chain 0.18 with one block, 0.21 with 16; ResNet-152 step (1652 kernels, 2020
// periods) 3.7 / 3.1 / 2.9 with 1 / 8 / 16; four ViT-H steps (6692 kernels, 13 875 periods) do not fit fewer than 16.  A block
// more takes work off the others' lanes in every iteration, an exchange costs 500-700 cycles whatever the size: one block only
// where there is next to nothing to share (E bounds the periods).
// (0: none can be placed)
int plan_chip_blocks(int64_t E, bool several, bool cyclic)
{
    const int most = chip_largest(cyclic ? kOneCycle : kOnePlan);
    return E <= 1024 && !several && most > 1 ? 1 : most;
}
int plan_batch_most_blocks() { return chip_largest(kManyPlans); }

// Worth launching (0: no; 1: the device decides, from the number of periods that it counted; 2: fits whatever their number).
int plan_chip_possible(int64_t K, int64_t E, int C, bool host_cap, bool cyclic)
{
    if (E < 1 || C < 1 || K > kChipMaxSlots || (cyclic ? 2 * K : K) >= (int64_t)kSlotTop) return 0;
    const int64_t room = chip_smem_budget(cyclic ? kOneCycle : kOnePlan), most = (E + C - 1) / C;
    if (most <= kChipMaxPeriods && (int64_t)chip_smem_core(K, most, C, host_cap, cyclic) <= room) return 2;
    return (int64_t)chip_smem_core(K, most < 64 ? most : 64, C, host_cap, cyclic) <= room ? 1 : 0;
}

// alone: no other planner is queued behind (plan_chip_possible == 2).  cyclic (steady-state planning): A.start is the unrolled clock [2K + 1], the period and geometry arrays hold unrolled slots.
cudaError_t launch_plan_chip(const PlanArgs &A, const Workspace &w, int C, bool cyclic, bool alone, cudaStream_t s)
{
    const int which = cyclic ? kOneCycle : kOnePlan;
    BatchArgs B;
    B.variants = nullptr; B.P0 = nullptr; B.P_out = nullptr; B.host_cap = 0;
    ChipArgs O = chip_args(which, w);
    O.alone = alone ? 1 : 0;
    return launch_chip(which, A, O, B, 1, C, s);
}

// ---------------------------------------------------------------------------------------------
// Batch: a cluster per variant, then one block per variant for the stability pairs.
// ---------------------------------------------------------------------------------------------
// stability[v] = (|M_v & M_0|, |M_v | M_0|) over the migrated periods of variant v and of variant 0; (-1, -1) if
// either plan is missing.  Also folds the call-wide status word (trace validation) into every variant's summary[7].
__global__ void __launch_bounds__(256) k_batch_finish(int64_t Pn_bound, const int64_t *Pn_dev, const g10_migration *out, int64_t out_cap,
                                                      int64_t *summary, int64_t *stability, const ull *status)
{
    extern __shared__ unsigned s_bits[];
    __shared__ int s_inter;
    const int v = blockIdx.x;
    const int64_t Pn = *Pn_dev < Pn_bound ? *Pn_dev : Pn_bound;
    const int words = (int)((Pn + 31) / 32);
    const int64_t n0 = summary[0] < out_cap ? summary[0] : out_cap, nv = summary[v * 8] < out_cap ? summary[v * 8] : out_cap;
    const bool ok = summary[2] >= 0 && summary[v * 8 + 2] >= 0;
    if (threadIdx.x == 0) s_inter = 0;
    for (int j = threadIdx.x; j < words; j += blockDim.x) s_bits[j] = 0;
    __syncthreads();
    if (ok) {
        for (int64_t j = threadIdx.x; j < n0; j += blockDim.x) { const int p = out[j].period; atomicOr(&s_bits[p >> 5], 1u << (p & 31)); }
        __syncthreads();
        int mine = 0;
        const g10_migration *mv = out + (size_t)v * out_cap;
        for (int64_t j = threadIdx.x; j < nv; j += blockDim.x) { const int p = mv[j].period; mine += (s_bits[p >> 5] >> (p & 31)) & 1u; }
        mine = __reduce_add_sync(0xffffffffu, mine);
        if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&s_inter, mine);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        stability[2 * v] = ok ? s_inter : -1;
        stability[2 * v + 1] = ok ? n0 + nv - s_inter : -1;
        summary[v * 8 + 7] |= (int64_t)*status;
    }
}

int batch_max_periods()          // periods whose bitmap fits the finishing kernel's shared memory
{
    return 200 * 1024 * 8;
}

static cudaError_t run_batch_finish(int64_t geo_stride, const int64_t *Pn_dev, const g10_migration *mig, int64_t out_cap, int64_t *summary,
                                    int V, int64_t *stability, const ull *status_word, cudaStream_t s)
{
    const int64_t bound = geo_stride < batch_max_periods() ? geo_stride : batch_max_periods();
    const size_t smem = (size_t)((bound + 31) / 32) * 4;
    cudaError_t e = allow_any<k_batch_finish>();
    if (e != cudaSuccess) return e;
    k_batch_finish<<<V, 256, smem, s>>>(bound, Pn_dev, mig, out_cap, summary, stability, status_word); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_batch_finish(const DeviceTrace &t, const Workspace &w, const PlanParams &p, int V, int64_t *stability, const ull *status_word,
                                cudaStream_t s)
{
    return run_batch_finish(t.E > 0 ? t.E : 1, w.counts + 1, p.migrations, p.migrations_cap, p.summary, V, stability, status_word, s);
}

cudaError_t launch_plan_batch(const PlanArgs &A, const Workspace &w, int V, int C, const BatchArgs &B, int64_t *stability, cudaStream_t s)
{
    ChipArgs O = chip_args(kManyPlans, w);
    O.busy_global = nullptr; O.hocc_global = nullptr;      // (the workspace has no room per variant)
    cudaError_t e = launch_chip(kManyPlans, A, O, B, V, C, s);
    if (e != cudaSuccess) return e;
    return run_batch_finish(A.geo_stride, A.Pn_dev, A.out, A.out_cap, A.summary, V, stability, A.status, s);
}

}  // namespace g10
