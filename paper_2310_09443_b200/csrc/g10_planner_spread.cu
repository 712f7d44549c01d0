// Algorithm 1 for long timelines whose state fits the shared memory of the whole GPU (148 SMs, 32 MB: a million slots and a
// million periods): the lazy evaluation of g10_planner_lazy.cu with every piece of hot state in some SM's shared memory.
//   - The timeline is cut into tiles of 64 slots, tile t in block t mod G: pressure above capacity per slot; smallest and largest
//     value, a pending offset and the total duration per tile.  A range of slots, however long, is thus spread evenly over all
//     blocks, and so are the tiles near capacity, which cluster.
//   - Period p is kept by block p mod G, in 16 bytes: rounded score, inactive and absent slots, destination, and whether the score is
//     FRESH (exact) or a bound (pressure only falls, so an earlier score is one).
// Per iteration:
//  A  every block applies the last commit to its tiles, compares its periods with it (absent ranges that meet: no longer FRESH;
//     transfer windows on the same channel that meet: is the destination still possible?  Channels only fill up: SSD -> host ->
//     erased) and publishes its best FRESH score and its eight best bounds; grid barrier;
//  R  rounds: the published bounds that may beat the best exact score are rescored by all blocks together, each over its own
//     tiles, with the shares added into grid-wide sums; grid barrier; the best exact score is updated.  A block whose published
//     bounds are used up while the last may still beat the best score publishes more;
//  D  no bound left that may beat it: commit.
// All decisions are taken from data every block has, so the control flow is the same in every block.  Rounded scores steer the
// search; anything within kNear of a decision is settled by exact 128-bit comparison.
// What bounds it: a chain of block-wide phases, 28 us an iteration on a million kernels, 0.40 s for the plan.  When it was 70 k cycles
// the pass over the periods took 14 k, rescoring 27 k (1.45 rounds of 230 periods each), the choice of what to rescore 8 k (less since),
// 2.7 grid barriers 15 k with the wait for the slowest block.  With slots and periods in global memory (g10_planner_lazy.cu) an
// iteration reads 140 MB through the L2: 0.97 s for the plan.  Durations are read from global memory when a tile is sorted or a range's end scored: in
// shared memory they cost 4 bytes a slot and saved nothing.
#include "g10_planner.cuh"

namespace g10 {

constexpr int kSpTile = 64;                     // slots per tile
constexpr int kSpRound = 512;                   // periods rescored together, at most
constexpr int kSpEdge = 2 * kSpRound;           // pairs in which the period covers the tile in part
constexpr int kSpSort = 12;                     // tiles sorted together (one warp each; a round has about four in a block)
constexpr int kSpDirect = 2 * kPlanWarps;       // up to this many (period, tile) pairs are read slot by slot rather than sorted
constexpr float kFirst = 0.97f;                 // the first round takes bounds down to this share of the best one (0.6 to 0.998: the same time)
// Bounds below kLikely of the lowest of the last kSpPast winners are not listed at first.  (Scores go up and down from winner to winner:
// with the last one alone every third iteration had to publish again, with four every hundredth; eight winners or 0.6 list more than
// they spare.)
constexpr float kLikely = 0.8f;
constexpr int kSpPast = 4;
constexpr double kNear = 1e-6;                  // (scores are kept as floats, rounded up: 2^-23)
constexpr int kSpTop = 8;                       // bounds a block publishes
constexpr int kSpSeg = 32;                      // likely bounds a warp may list (one per lane when they are ranked)
constexpr int kSpPool = kLazyMaxBlocks * kSpTop;
static_assert(kPlanWarps == 16, "two chunks of warp counts per 32 lanes");
static_assert(kSpRound == kPlanThreads, "one thread per period of a round");
constexpr int kSpLimbs = 4;                     // a benefit (below 2^84) as 21-bit limbs

// What a block tells the grid: its best exactly scored period, its best bounds (descending; anything it did not list is no larger
// than the last), its largest pressure above capacity.
struct __align__(16) SpProp {
    ull ben_lo, ben_hi, cost;
    int idx;                                    // period << 1 | destination, -1 = none
    unsigned key;                               // its rounded score
    unsigned skey[kSpTop];
    int sidx[kSpTop];                           // period << 1 | destination, -1 = none
    long long peak;
};
static_assert(sizeof(SpProp) % 16 == 0 && 2 * sizeof(LazyProp) >= sizeof(SpProp), "workspace for two LazyProp a block");

struct SpreadArgs {
    ull *c_ben_lo, *c_ben_hi, *c_cost;          // [periods] last computed benefit (exact or a bound), cost of the current destination
    SpProp *props;                              // [2][kLazyMaxBlocks]
    ull *partials;                              // [3][2][kSpRound] sums of the low 44 bits and of the rest (three buffers in turn)
    unsigned *flag;                             // raised by a block that cannot keep its part (a duration of 2^32 ns or more)
    unsigned *done;                             // set to 1 when this kernel produced the plan
    int smem_bytes;
};

// A period: x = score (float bits, rounded up; 0 = no benefit), inactive slots [a, b] and absent slots [ap, bp] of the current
// destination (21 bits each), destination + 1 (0 = erased), FRESH.  a, b and ap head a word each: the pass over all periods compares
// the words as they are.
struct SpPeriod { int a, b, ap, bp, dest; bool fresh; };
constexpr unsigned kSpFresh = 4u, kSpDest = 3u;
__device__ __forceinline__ uint4 sp_pack(unsigned key, int a, int b, int ap, int bp, int dest, bool fresh)
{
    return make_uint4(key, (unsigned)a << 11 | (unsigned)bp >> 10, (unsigned)b << 11 | ((unsigned)bp & 0x3ffu), (unsigned)ap << 11 | (fresh ? kSpFresh : 0u) | (unsigned)(dest + 1));
}
__device__ __forceinline__ int sp_bp(uint4 q) { return (int)((q.y & 0x7ffu) << 10 | (q.z & 0x3ffu)); }
__device__ __forceinline__ SpPeriod sp_unpack(uint4 q)
{
    SpPeriod r;
    r.a = (int)(q.y >> 11); r.b = (int)(q.z >> 11); r.ap = (int)(q.w >> 11); r.bp = sp_bp(q);
    r.dest = (int)(q.w & kSpDest) - 1; r.fresh = (q.w & kSpFresh) != 0u;
    return r;
}
constexpr int kSpMaxSlots = (1 << 21) - 1;

__device__ __forceinline__ unsigned sp_key(u128 ben, ull cost)
{
    if (ben == 0) return 0u;
    Cand c;
    c.ben = ben; c.cost = cost; c.idx = 0; c.dest = 0;
    return __float_as_uint(__double2float_ru(cand_key(c) * (1.0 + 1e-14)));     // (positive floats compare like integers)
}
__device__ __forceinline__ double sp_val(unsigned key) { return (double)__uint_as_float(key); }

// Rounded scores above `hi` beat the best exact score, those below `lo` do not; what is between is settled exactly.
struct SpBar { unsigned lo, hi; };
__device__ __forceinline__ SpBar sp_bar(const Cand &t)
{
    if (t.idx < 0) return {1u, 0u};
    const double k = cand_key(t);
    return {__float_as_uint(__double2float_rd(k * (1.0 - kNear))), __float_as_uint(__double2float_ru(k * (1.0 + kNear)))};
}
// Could a period with rounded score `key` (an upper bound) beat t?
__device__ __forceinline__ bool sp_may_beat(const SpreadArgs &S, int p, unsigned key, SpBar bar, const Cand &t)
{
    if (key < bar.lo) return false;
    if (key > bar.hi) return true;
    Cand x;
    x.ben = ((u128)__ldcg(&S.c_ben_hi[p]) << 64) | __ldcg(&S.c_ben_lo[p]); x.cost = __ldcg(&S.c_cost[p]); x.idx = p; x.dest = 0;
    return cand_beats(x, t);
}

// A tile's slots in order of their pressure, for the periods of a round that cover it all and find some of its slots less than their
// size above capacity: with prefix sums of the durations and of pressure x duration, a period's benefit is a binary search
// instead of 64 slots (a round's periods mostly overlap: the same few tiles near capacity are wanted a hundred times).
struct __align__(16) SpSorted {
    long long v[kSpTile];                       // pressure above capacity, at least 0 and at most 2^40 (tensors are smaller), ascending
    ull lo[kSpTile + 1], hi[kSpTile + 1];       // sums of (v mod 2^20) x duration and of (v >> 20) x duration over the first n
    unsigned d[kSpTile + 1];                    // sums of the durations (a tile's total is below 2^32 ns)
    int n, lt, pad;
};

// Where a block's dynamic shared memory goes: byte offsets of its arrays, and what they take together (the same function measures
// and lays out, so that a trace is never taken on that the arrays have no room for).
struct SpreadLayout {
    // (tiles: of slots, a block, at most; runs: of 32 periods, likewise)
    size_t mm;                                  // [tiles] longlong2
    size_t hot;                                 // [runs * 32] uint4
    size_t r_acc, r_s, r_e, r_ap, r_bp;         // a round: [kSpLimbs][kSpRound] unsigned; [kSpRound] long long, int, int, int
    size_t edge;                                // [kSpEdge] unsigned
    size_t sorted;                              // [kSpSort] SpSorted
    size_t mid, full;                           // [tiles] unsigned, ull
    size_t pkey, pidx, pdone;                   // [kSpTop * G] unsigned, int, unsigned char
    size_t ex;                                  // [tiles * kSpTile] long long
    size_t off, tsum;                           // [tiles] long long, unsigned
    size_t total;
};
__host__ __device__ inline SpreadLayout spread_layout(int64_t K, int64_t Pn, int G)
{
    SpreadLayout l;
    size_t at = 0;
    auto take = [&](size_t bytes) { const size_t p = at; at += (bytes + 15) / 16 * 16; return p; };
    const size_t tiles = (size_t)(((K + kSpTile - 1) / kSpTile + G - 1) / G), runs = (size_t)(((Pn + G - 1) / G + 31) / 32);
    l.mm = take(tiles * 16);
    l.hot = take(runs * 32 * 16);
    l.r_acc = take((size_t)kSpRound * 4 * kSpLimbs);
    l.r_s = take((size_t)kSpRound * 8); l.r_e = take((size_t)kSpRound * 4);
    l.r_ap = take((size_t)kSpRound * 4); l.r_bp = take((size_t)kSpRound * 4);
    l.edge = take((size_t)kSpEdge * 4);
    l.sorted = take(kSpSort * sizeof(SpSorted));
    l.mid = take(tiles * 4); l.full = take(tiles * 8);
    l.pkey = take((size_t)G * kSpTop * 4); l.pidx = take((size_t)G * kSpTop * 4); l.pdone = take((size_t)G * kSpTop);
    l.ex = take(tiles * kSpTile * 8);
    l.off = take(tiles * 8); l.tsum = take(tiles * 4);
    l.total = at;
    return l;
}

__global__ void __launch_bounds__(kPlanThreads, 1) k_plan_spread(PlanArgs A, SpreadArgs S)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    __shared__ Cand s_cand[kPlanWarps + 1];
    __shared__ BestScratch s_best;
    __shared__ long long s_max[kPlanWarps + 1];
    __shared__ unsigned s_tk[kSpTop], s_fk[kPlanWarps], s_wm[kPlanWarps];
    __shared__ uint2 s_seg[kPlanWarps][kSpSeg];                                 // score, period << 1 | destination
    __shared__ int s_ti[kSpTop], s_cnt[kPlanWarps];
    constexpr int kChunks = (kSpPool + kPlanThreads - 1) / kPlanThreads;        // entries of the pool a thread looks at
    __shared__ Cand s_fin[32];
    __shared__ int s_nfin, s_nmid, s_nedge;
    __shared__ Cand s_one;
    __shared__ ull s_full[32];                                                  // [group of 32 tiles]
    __shared__ unsigned char s_refresh[kLazyMaxBlocks];
    if (*S.done) return;                                     // (same answer in every thread of the grid: written by an earlier launch)
    const int G = gridDim.x, c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t Pn64 = *A.Pn_dev < A.geo_stride ? *A.Pn_dev : A.geo_stride;
    if (A.K < 1 || A.K > kSpMaxSlots || Pn64 > 0x3fffffff) return;               // (the same answer in all blocks)
    const SpreadLayout l = spread_layout(A.K, Pn64, G);
    if (l.total > (size_t)S.smem_bytes) return;                                 // (here too)
    const int K = (int)A.K, Pn = (int)Pn64;
    const int64_t limit = (A.max_iterations <= 0 || A.max_iterations > Pn64) ? Pn64 : A.max_iterations;
    const int NT = (K + kSpTile - 1) / kSpTile;
    const int my_tiles = NT > c ? (NT - c + G - 1) / G : 0, my_runs = Pn > c ? ((Pn - c + G - 1) / G + 31) / 32 : 0;
    longlong2 *mm = (longlong2 *)(s_raw + l.mm);                                // [tiles] smallest / largest, offset included
    uint4 *hot = (uint4 *)(s_raw + l.hot);
    unsigned *r_acc = (unsigned *)(s_raw + l.r_acc);                            // [limb][period] (sums of far fewer than 2^11 limbs)
    long long *r_s = (long long *)(s_raw + l.r_s);
    int *r_e = (int *)(s_raw + l.r_e);                                          // pool entry
    int *r_ap = (int *)(s_raw + l.r_ap), *r_bp = (int *)(s_raw + l.r_bp);
    unsigned *s_edge = (unsigned *)(s_raw + l.edge);                            // period of the round << 20 | local tile
    SpSorted *sorted = (SpSorted *)(s_raw + l.sorted);
    unsigned *t_mid = (unsigned *)(s_raw + l.mid);                              // tiles of a round that are near capacity
    ull *t_full = (ull *)(s_raw + l.full);                                      // duration of the tiles of this group of 32 so far that are above it for every period of the round
    unsigned *pkey = (unsigned *)(s_raw + l.pkey);                              // published bounds, [rank in the list][block]
    int *pidx = (int *)(s_raw + l.pidx);                                        // period << 1 | destination, -1 = none
    unsigned char *pdone = s_raw + l.pdone;
    long long *ex = (long long *)(s_raw + l.ex);
    long long *off = (long long *)(s_raw + l.off);
    unsigned *tsum = (unsigned *)(s_raw + l.tsum);
    auto owner_entry = [&](int p) { return p % G == c ? p / G : -1; };

    unsigned gen = 0;
    int64_t n_mig = 0, rounds = 0, bytes_ssd = 0, bytes_host = 0;
    int status = -1;
    long long peak = 0;
    int pbuf = 0, pp = 0;

    // ---- own slots, tiles and periods
    bool bad = false;
    for (int x = tid; x < my_tiles * kSpTile; x += kPlanThreads) {
        const int64_t k = ((int64_t)(x / kSpTile) * G + c) * kSpTile + x % kSpTile;
        ex[x] = k < K ? A.P[k] - A.cap : 0;
    }
    for (int lt = tid; lt < my_tiles; lt += kPlanThreads) {
        const int t = lt * G + c;
        const long long d = A.start[t * kSpTile + kSpTile < K ? t * kSpTile + kSpTile : K] - A.start[t * kSpTile];
        if (d >> 32) bad = true;
        off[lt] = 0; tsum[lt] = (unsigned)d;
    }
    if (c == 0) for (int j = tid; j < 3 * kSpRound * 2; j += kPlanThreads) S.partials[j] = 0;
    __syncthreads();
    // smallest and largest value of local tile lt (one warp)
    auto refresh_tile = [&](int lt) {
        const int t = lt * G + c, n = K - t * kSpTile < kSpTile ? K - t * kSpTile : kSpTile;
        long long mn = 0x7fffffffffffffffll, mx = -0x7fffffffffffffffll - 1;
#pragma unroll
        for (int j = 0; j < kSpTile; j += 32)
            if (j + lane < n) {
                const long long v = ex[lt * kSpTile + j + lane];
                mn = v < mn ? v : mn; mx = v > mx ? v : mx;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long a = __shfl_xor_sync(0xffffffffu, mn, o), b = __shfl_xor_sync(0xffffffffu, mx, o);
            mn = a < mn ? a : mn; mx = b > mx ? b : mx;
        }
        if (lane == 0) mm[lt] = make_longlong2(mn + off[lt], mx + off[lt]);
    };
    for (int lt = warp; lt < my_tiles; lt += kPlanWarps) refresh_tile(lt);
    // (re)starts a period on destination X: its first bound is the benefit it would have if its whole absent range were at least s
    // above capacity
    auto begin_period = [&](int p, int e, int X, int a, int b) {
        const int ap = A.geo_a[X * A.geo_stride + p], bp = A.geo_b[X * A.geo_stride + p];
        const u128 ben = (u128)(ull)A.bytes[A.per_t[p]] * (u128)(ull)(A.start[bp + 1] - A.start[ap]);
        const ull cost = 2ull * (ull)A.geo_t[X * A.geo_stride + p];
        S.c_ben_lo[p] = (ull)ben; S.c_ben_hi[p] = (ull)(ben >> 64); S.c_cost[p] = cost;
        hot[e] = sp_pack(sp_key(ben, cost), a, b, ap, bp, X, false);
    };
    for (int e = tid; e < my_runs * 32; e += kPlanThreads) {
        const int64_t p = (int64_t)e * G + c;
        hot[e] = make_uint4(0, 0, 0, 0);
        if (p >= Pn) continue;
        // nothing is booked yet: the first usable destination it is
        const bool room = A.host_capacity == 0 || (uint64_t)A.bytes[A.per_t[p]] <= A.host_capacity;
        const int X = A.geo_a[p] >= 0 ? 0 : A.geo_a[A.geo_stride + p] >= 0 && room ? 1 : -1;
        if (X >= 0) begin_period((int)p, e, X, A.per_u[p] + 1, A.per_v[p] - 1);
    }
    if (bad) atomicOr(S.flag, 1u);
    __syncthreads();
    if (!grid_barrier(A.bar, G, gen)) status = -2;
    else if (__ldcg(S.flag) != 0u) return;                   // (nothing changed: the planner queued behind this one takes over)

    struct { int idx, dest, a, ap, bp, b; int64_t s, t, t_r, t_end; } w = {-1, -1, 0, 0, -1, -1, 0, 0, 0, 0};     // the pending commit
    unsigned likely = 0;                                     // bounds below this are not listed at first
    float last_key = 0.0f, won[kSpPast] = {};                // the last winner's score, and those of the last few
    bool pending = false;
    Cand gBest;                                              // best exactly scored period known to the grid
    gBest.ben = 0; gBest.cost = 1; gBest.idx = -1; gBest.dest = -1;

    // One pass of the block over its periods.  With `classify` the pending commit is applied to them first (its bookings are not in
    // A.busy yet).  With a floor only bounds that may beat it are listed.  Publishes into buffer pbuf.
    auto scan = [&](bool classify, bool with_floor) {
        unsigned fk = 0, f2 = 0;                                    // the lane's two largest exact scores
        int fe = -1, n = 0;                                         // entry of the largest; bounds listed by this warp
        const int64_t *bo = A.busy + (size_t)(2 * (w.dest < 0 ? 0 : w.dest)) * A.K, *bi = bo + A.K;
        const SpBar bar = sp_bar(gBest);
        const unsigned least = with_floor ? bar.lo : likely ? likely : 1u;
        const unsigned w_tag = (unsigned)(w.dest + 1), w_ap = (unsigned)w.ap << 11, w_a1 = (unsigned)(w.a + 1) << 11, w_bp1 = (unsigned)(w.bp + 1) << 11;
        const bool host_fills = A.host_capacity != 0 && w.dest == G10_DEST_HOST;
        if (tid == 0) s_nfin = 0;
        if (tid < kSpTop) { s_tk[tid] = 0u; s_ti[tid] = -1; }
        auto list = [&](bool take, uint4 q, int p) {
            const unsigned m = __ballot_sync(0xffffffffu, take);
            if (m == 0u) return;
            const int pos = n + __popc(m & ((1u << lane) - 1u));
            if (take && pos < kSpSeg) s_seg[warp][pos] = make_uint2(q.x, (unsigned)p << 1 | ((q.w & kSpDest) - 1u));
            n += __popc(m);
        };
        auto look = [&](uint4 q, int e) {
            const int p = e * G + c;
            const bool exact = (q.w & kSpFresh) != 0u;
            if (exact) { f2 = q.x > fk ? fk : q.x > f2 ? q.x : f2; fe = q.x > fk ? e : fe; fk = q.x > fk ? q.x : fk; }
            bool take = !exact & (q.x >= least);
            if (with_floor && take) take = sp_may_beat(S, p, q.x, bar, gBest);
            list(take, q, p);
        };
        // (a short loop, the next run's periods on the way: unrolled four times it took longer, for its instructions)
        unsigned touched = 0;                                       // (the warp has at most 32 runs)
        uint4 next = warp < my_runs ? hot[warp * 32 + lane] : make_uint4(0, 0, 0, 0);
#pragma unroll 1
        for (int r = warp, n_run = 0; r < my_runs; r += kPlanWarps, ++n_run) {
            const int e = r * 32 + lane;
            uint4 q = next;
            if (r + kPlanWarps < my_runs) next = hot[e + kPlanWarps * 32];
            if (classify) {
                // does the commit concern the period at all?  Its channel windows meet those of the commit (rarely: these runs come
                // after the others); an exact score's absent range meets it
                // (out: a < w.ap and w.a < ap; in: bp < w.b and w.bp < b)
                const int bp = sp_bp(q);
                bool meets = ((q.w & kSpDest) == w_tag) & (((q.y < w_ap) & (q.w >= w_a1)) | ((q.z >= w_bp1) & (bp < w.b)));     // (no branches)
                if (host_fills) meets = meets || ((q.w & kSpDest) == G10_DEST_HOST + 1 && q.y >> 11 <= (unsigned)w.b && (unsigned)w.a <= q.z >> 11);
                const bool stale = ((q.w & kSpFresh) != 0u) & (q.w < w_bp1) & (w.ap <= bp);
                if (stale) { q.w &= ~kSpFresh; hot[e].w = q.w; }
                if (__any_sync(0xffffffffu, meets)) { touched |= 1u << n_run; continue; }
            }
            look(q, e);
        }
        if (classify) {
            __syncwarp();
#pragma unroll 1
            while (touched) {
                const int r = warp + (__ffs(touched) - 1) * kPlanWarps, e = r * 32 + lane, p = e * G + c;
                touched &= touched - 1;
                const SpPeriod P = sp_unpack(hot[e]);
                const bool meet_out = P.dest == w.dest && P.a < w.ap && w.a < P.ap, meet_in = P.dest == w.dest && P.bp < w.b && w.bp < P.b;
                bool lost = false;
                if (meet_out || meet_in) {
                    const int64_t tq = (int64_t)(S.c_cost[p] >> 1), q_r = A.start[P.a], q_end = A.start[P.b + 1];
                    lost = (meet_out && window_conflict<false, true>(A.start, bo, w.a, w.ap - 1, w.t_r, w.t_r + w.t, q_r, q_r + tq, P.a, P.ap - 1)) ||
                           (meet_in && window_conflict<false, true>(A.start, bi, w.bp + 1, w.b, w.t_end - w.t, w.t_end, q_end - tq, q_end, P.bp + 1, P.b));
                }
                // host memory of these slots has filled up (finite capacity): is there still room?
                const bool room = host_fills && P.dest == G10_DEST_HOST && P.a <= w.b && w.a <= P.b;
                unsigned todo = __ballot_sync(0xffffffffu, lost || room);
                __syncwarp();
#pragma unroll 1
                while (todo) {                              // the whole warp, one period after the other
                    const int src = __ffs(todo) - 1;
                    todo &= todo - 1;
                    const int e2 = r * 32 + src, p2 = e2 * G + c;
                    const bool gone = __shfl_sync(0xffffffffu, lost, src);
                    const SpPeriod Q = sp_unpack(hot[e2]);
                    const int64_t s2 = A.bytes[A.per_t[p2]];
                    auto host_room = [&]() {
                        if (A.host_capacity == 0) return true;
                        bool ok = true;
                        for (int k = Q.a + lane; k <= Q.b; k += 32) {
                            const uint64_t more = w.dest == G10_DEST_HOST && k >= w.a && k <= w.b ? (uint64_t)w.s : 0u;
                            if ((uint64_t)__ldcg(&A.hocc[k]) + more + (uint64_t)s2 > A.host_capacity) ok = false;
                        }
                        return __all_sync(0xffffffffu, ok) != 0;
                    };
                    if (!gone && host_room()) continue;
                    // SSD -> host -> erased.  (A period that leaves the SSD does so because of a commit to the SSD: nothing is pending
                    // on the host's channels.)
                    bool to_host = false;
                    if (Q.dest == G10_DEST_SSD) {
                        const int ap = A.geo_a[A.geo_stride + p2];
                        if (ap >= 0) {
                            const int bp = A.geo_b[A.geo_stride + p2];
                            const int64_t t2 = A.geo_t[A.geo_stride + p2], q_r = A.start[Q.a], q_end = A.start[Q.b + 1];
                            to_host = window_free(A, A.busy + (size_t)(2 * G10_DEST_HOST) * A.K, q_r, q_r + t2, Q.a, ap - 1, lane) &&
                                      window_free(A, A.busy + (size_t)(2 * G10_DEST_HOST + 1) * A.K, q_end - t2, q_end, bp + 1, Q.b, lane) && host_room();
                        }
                    }
                    if (lane == 0) { if (to_host) begin_period(p2, e2, G10_DEST_HOST, Q.a, Q.b); else hot[e2] = make_uint4(0, 0, 0, 0); }
                }
                __syncwarp();
                look(hot[e], e);
            }
        }
        long long top = -0x7fffffffffffffffll - 1;                  // largest pressure above capacity of the own tiles
        for (int lt = tid; lt < my_tiles; lt += kPlanThreads) { const long long v = mm[lt].y; top = v > top ? v : top; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { const long long y = __shfl_xor_sync(0xffffffffu, top, o); top = y > top ? y : top; }
        const unsigned wf = __reduce_max_sync(0xffffffffu, fk);
        __syncwarp();
        uint2 mine = lane < n ? s_seg[warp][lane] : make_uint2(0, 0);
        if (const unsigned m = __reduce_max_sync(0xffffffffu, mine.x); lane == 0) { s_fk[warp] = wf; s_wm[warp] = m; s_max[warp] = top; s_cnt[warp] = n; }
        __syncthreads();
        // the exactly scored periods that may be the best of them (their scores are on the way while the bounds are ranked)
        auto exact = [&](int p) {
            Cand x;
            x.ben = ((u128)S.c_ben_hi[p] << 64) | S.c_ben_lo[p]; x.cost = S.c_cost[p]; x.idx = p;
            x.dest = (int)(hot[owner_entry(p)].w & kSpDest) - 1;
            return x;
        };
        const unsigned bf = __reduce_max_sync(0xffffffffu, lane < kPlanWarps ? s_fk[lane] : 0u);
        const unsigned thr = bf ? __float_as_uint((float)(sp_val(bf) * (1.0 - kNear))) : 0u;
        if (wf != 0u && wf >= thr) {
            if (!__any_sync(0xffffffffu, f2 >= thr)) {
                if (fk >= thr) { const int x = atomicAdd(&s_nfin, 1); if (x < 32) s_fin[x] = exact(fe * G + c); }
            } else
#pragma unroll 1
                for (int r = warp; r < my_runs; r += kPlanWarps) {
                    const uint4 q = hot[r * 32 + lane];
                    if (q.x >= thr && (q.w & kSpFresh)) { const int x = atomicAdd(&s_nfin, 1); if (x < 32) s_fin[x] = exact((r * 32 + lane) * G + c); }
                }
        }
        // more bounds than the lists hold: the lowest score that at least kSpTop of them reach and the lists hold, by bisection (if too
        // many share one score, any of those: what is not listed is no larger than what is).  Under a floor only bounds that may beat it
        // count, here as above: with those that share its score but lose the exact comparison the lists could be full of bounds that
        // nobody rescores, publication after publication.
        auto counts = [&](uint4 q, int p) { return !(q.w & kSpFresh) && (!with_floor || sp_may_beat(S, p, q.x, bar, gBest)); };
        if (__any_sync(0xffffffffu, lane < kPlanWarps && s_cnt[lane] > kSpSeg)) {
            unsigned lo = least, hi = 0x7f800000u;                  // too many; too few (or just right, which ends the search)
            bool fits = false;
#pragma unroll 1
            while (!fits && hi - lo > 1u) {
                const unsigned mid = lo + (hi - lo) / 2;
                unsigned m = 0;
#pragma unroll 1
                for (int r = warp; r < my_runs; r += kPlanWarps) { const uint4 q = hot[r * 32 + lane]; m += q.x >= mid && counts(q, (r * 32 + lane) * G + c) ? 1u : 0u; }
                m = __reduce_add_sync(0xffffffffu, m);
                __syncthreads();
                if (lane == 0) s_cnt[warp] = (int)m;
                __syncthreads();
                const unsigned z = lane < kPlanWarps ? (unsigned)s_cnt[lane] : 0u;
                const bool many = __reduce_max_sync(0xffffffffu, z) > (unsigned)kSpSeg;
                if (many) lo = mid;
                else { hi = mid; fits = __reduce_add_sync(0xffffffffu, z) >= (unsigned)kSpTop; }
            }
            n = 0;
#pragma unroll 1
            for (int pass = 0; pass < (fits ? 1 : 2); ++pass)
#pragma unroll 1
                for (int r = warp; r < my_runs; r += kPlanWarps) {
                    const uint4 q = hot[r * 32 + lane];
                    list((pass == 0 ? q.x >= hi : q.x == lo) && counts(q, (r * 32 + lane) * G + c), q, (r * 32 + lane) * G + c);
                }
            __syncwarp();
            mine = lane < n ? s_seg[warp][lane] : make_uint2(0, 0);
            const unsigned m = __reduce_max_sync(0xffffffffu, mine.x);
            __syncthreads();
            if (lane == 0) s_wm[warp] = m;
            __syncthreads();
        }
        // the best kSpTop of the listed ones.  The kSpTop-th largest of the warps' maxima bounds them from below; of the few that
        // reach it everyone counts how many come before its own
        {
            const unsigned v = lane < kPlanWarps ? s_wm[lane] : 0u;
            int before = 0;
#pragma unroll
            for (int j = 0; j < kPlanWarps; ++j) { const unsigned y = __shfl_sync(0xffffffffu, v, j); before += y > v || (y == v && j < lane) ? 1 : 0; }
            const unsigned at = __ballot_sync(0xffffffffu, before == kSpTop - 1);
            const unsigned t = __shfl_sync(0xffffffffu, v, __ffs(at) - 1);              // (0 if fewer warps list any)
            const bool keep = mine.x != 0u && mine.x >= t;
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (keep) s_seg[warp][__popc(m & ((1u << lane) - 1u))] = mine;
            if (lane == 0) s_cnt[warp] = __popc(m);
            __syncthreads();
            if (keep) {
                int rank = 0;
#pragma unroll 1
                for (int u = 0; u < kPlanWarps; ++u)
#pragma unroll 1
                    for (int j = 0, z = s_cnt[u]; j < z; ++j) { const uint2 q = s_seg[u][j]; rank += q.x > mine.x || (q.x == mine.x && q.y < mine.y) ? 1 : 0; }
                if (rank < kSpTop) { s_tk[rank] = mine.x; s_ti[rank] = (int)mine.y; }
            }
        }
        __syncthreads();
        Cand best;
        best.ben = 0; best.cost = 1; best.idx = -1; best.dest = -1;
        const int n_fin = s_nfin;
        if (n_fin <= 32) {
            if (warp == 0) {
                if (lane < n_fin) best = s_fin[lane];
                if (n_fin > 1)
#pragma unroll 1
                    for (int o = 16; o > 0; o >>= 1) { const Cand y = cand_shfl_down(best, o); if (cand_beats(y, best)) best = y; }
            }
        } else {                                                    // very many close scores
#pragma unroll 1
            for (int r = warp; r < my_runs; r += kPlanWarps) {
                const uint4 q = hot[r * 32 + lane];
                if (q.x >= thr && (q.w & kSpFresh)) { const Cand y = exact((r * 32 + lane) * G + c); if (cand_beats(y, best)) best = y; }
            }
            best = block_best(best, s_cand);
        }
        SpProp &o = S.props[(size_t)pbuf * kLazyMaxBlocks + c];
        if (tid < kSpTop) { o.skey[tid] = s_tk[tid]; o.sidx[tid] = s_ti[tid]; }
        if (tid == 0) {
            o.ben_lo = (ull)best.ben; o.ben_hi = (ull)(best.ben >> 64); o.cost = best.cost; o.idx = best.idx < 0 ? -1 : best.idx << 1 | best.dest; o.key = best.idx < 0 ? 0u : hot[owner_entry(best.idx)].x;
        }
        if (warp == 1) {
            long long m = lane < kPlanWarps ? s_max[lane] : s_max[0];
#pragma unroll
            for (int z = 16; z > 0; z >>= 1) { const long long y = __shfl_xor_sync(0xffffffffu, m, z); m = y > m ? y : m; }
            if (lane == 0) o.peak = m;
        }
    };
    // The exactly best of the threads' candidates (at most one each, with its rounded score): the block's threads all get it.
    auto best_of = [&](const Cand &x, unsigned key) {
        const unsigned wk = __reduce_max_sync(0xffffffffu, key);
        if (lane == 0) s_fk[warp] = wk;
        __syncthreads();
        const unsigned m = __reduce_max_sync(0xffffffffu, lane < kPlanWarps ? s_fk[lane] : 0u);
        const bool near = key != 0u && sp_val(key) >= sp_val(m) * (1.0 - kNear);
        if (near) s_one = x;                                 // (usually one thread)
        if (m == 0u && tid == 0) s_one = x;
        if (__syncthreads_count(near) <= 1) return s_one;    // (nobody: thread 0's, which is none)
        return block_best_fast(x, &s_best, s_cand);
    };
    unsigned best_bound = 0;                                 // the largest published bound of the iteration
    // Reads publications of buffer `buf` into the pool of bounds (all, or those of the blocks that published again); returns the best
    // exactly scored one, and whether anything is above capacity.
    auto load = [&](int buf, bool only_flagged, bool *over) {
        Cand x;
        x.ben = 0; x.cost = 1; x.idx = -1; x.dest = -1;
        unsigned key = 0, bound = 0;
        bool above = false;
        for (int j = tid; j < G; j += kPlanThreads) {        // (G <= kPlanThreads: one block's values per thread)
            if (only_flagged && !s_refresh[j]) continue;
            const uint4 *src = (const uint4 *)&S.props[(size_t)buf * kLazyMaxBlocks + j];
            union { uint4 v[sizeof(SpProp) / 16]; SpProp o; } u;
#pragma unroll
            for (int q = 0; q < (int)sizeof(SpProp) / 16; ++q) u.v[q] = __ldcg(src + q);
            if (u.o.idx >= 0) { x.ben = ((u128)u.o.ben_hi << 64) | u.o.ben_lo; x.cost = u.o.cost; x.idx = u.o.idx >> 1; x.dest = u.o.idx & 1; key = u.o.key; }
            above = u.o.peak > 0;
            bound = u.o.skey[0];
#pragma unroll
            for (int q = 0; q < kSpTop; ++q) { pkey[q * G + j] = u.o.skey[q]; pidx[q * G + j] = u.o.sidx[q]; pdone[q * G + j] = 0; }
        }
        if (over != nullptr) {
            bound = __reduce_max_sync(0xffffffffu, bound);
            if (lane == 0) s_wm[warp] = bound;
            *over = __syncthreads_or(above) != 0;
            best_bound = __reduce_max_sync(0xffffffffu, lane < kPlanWarps ? s_wm[lane] : 0u);
        }
        const Cand b = best_of(x, key);
        __syncthreads();
        return b;
    };

#pragma unroll 1
    for (int64_t it = 0; status == -1; ++it) {
        bool barrier_since_booking = true;
        // ---------------- A: the pending commit on the own tiles: whole ones by their offset, the two at the ends slot by slot
        if (pending) {
            const int ta = w.ap / kSpTile, tb = w.bp / kSpTile;
            const int l0 = ta > c ? (ta - c + G - 1) / G : 0, l1 = tb >= c ? (tb - c) / G : -1;
#pragma unroll 1
            for (int lt = l0 + tid; lt <= l1; lt += kPlanThreads) {
                const int t = lt * G + c;
                if (t * kSpTile < w.ap || (t * kSpTile + kSpTile - 1 > w.bp && w.bp != K - 1)) continue;
                longlong2 m = mm[lt];
                m.x -= w.s; m.y -= w.s;
                mm[lt] = m; off[lt] -= w.s;
            }
#pragma unroll 1
            for (int end = 0; end < 2; ++end) {
                const int t = end ? tb : ta;
                if (t % G != c || (end && tb == ta) || warp != kPlanWarps - 1 - end) continue;
                if (!(t * kSpTile < w.ap || (t * kSpTile + kSpTile - 1 > w.bp && w.bp != K - 1))) continue;     // (a whole one)
                const int lt = t / G;
#pragma unroll
                for (int j = 0; j < kSpTile; j += 32) {
                    const int k = t * kSpTile + j + lane;
                    if (k >= w.ap && k <= w.bp) ex[lt * kSpTile + j + lane] -= w.s;
                }
                __syncwarp();
                refresh_tile(lt);
            }
            if (c == 0 && tid == 0) {
                if (n_mig - 1 < A.out_cap) {
                    g10_migration m;
                    m.period = w.idx; m.tensor = A.per_t[w.idx]; m.dest = w.dest; m.absent_first = w.ap; m.absent_last = w.bp;
                    m.iteration = (int32_t)(it - 1); m.evict_issue_ns = w.t_r; m.prefetch_issue_ns = w.t_end - w.t; m.transfer_ns = w.t;
                    A.out[n_mig - 1] = m;
                } else raise_status(A.status, G10_DEV_PLAN_OVERFLOW);
            }
        }
        if (pending && tid == 0) { const int e = owner_entry(w.idx); if (e >= 0) hot[e] = make_uint4(0, 0, 0, 0); }
        __syncthreads();
        scan(pending, false);
        if (!grid_barrier(A.bar, G, gen)) { status = -2; break; }
        bool over;
        gBest = load(pbuf, false, &over);
        pbuf ^= 1;
        if (A.fits_always || !over) { status = n_mig == 0 ? G10_ALREADY_FITS : G10_FIT; break; }
        if (it >= limit) { status = limit < Pn64 ? G10_ITERATION_LIMIT : G10_EXHAUSTED; break; }
        rounds += 1;
        if (pending) {
            if (c == 0) {
                book_winner(A, w.idx, w.dest);
                if (w.dest == G10_DEST_HOST && A.host_capacity != 0) for (int k = w.a + tid; k <= w.b; k += kPlanThreads) A.hocc[k] += w.s;
            }
            barrier_since_booking = false;
        }
        pending = false;
        // ---------------- R: rounds of joint rescoring
        // (compared: other blocks' periods, in the last choice; again_published: bounds were published again and none has been taken since)
        bool failed = false, compared = false, again_published = false;
        int round_no = 0;
        const int n_pool = G * kSpTop;
#pragma unroll 1
        for (;;) {
            const SpBar bar = sp_bar(gBest);
            // which published bounds are rescored now (the same choice in every block, in the same order): every unused one that
            // may beat the best exact score -- in the first round only those near the best bound (kFirst; the winner is usually
            // among them, and a strong exact score spares the rest)
            int msel;
            test_come_late(A.bar);
            {
                bool near = false;
                const unsigned floor0 = round_no == 0 ? __float_as_uint(fminf(__uint_as_float(best_bound), last_key > 0.0f ? last_key : __uint_as_float(best_bound)) * kFirst) : 0u;
                int mine = 0, at[kChunks];                    // the warp's, and for each of the thread's entries those before it in the warp (-1: not taken)
#pragma unroll
                for (int j = 0; j < kChunks; ++j) {
                    const int e = j * kPlanThreads + tid;
                    bool take = false;
                    if (e < n_pool && !pdone[e] && pidx[e] >= 0 && pkey[e] >= floor0) {
                        take = sp_may_beat(S, pidx[e] >> 1, pkey[e], bar, gBest);
                        near = near || (pkey[e] >= bar.lo && pkey[e] <= bar.hi);
                        if (!take) pdone[e] = 2;
                    }
                    const unsigned mk = __ballot_sync(0xffffffffu, take);
                    at[j] = take ? mine + __popc(mk & ((1u << lane) - 1u)) : -1;
                    mine += __popc(mk);
                }
                if (lane == 0) s_cnt[warp] = mine;
                // (other blocks' periods were compared exactly: see the barrier before the decision)
                compared = __syncthreads_or(near) != 0;
                const int v = lane < kPlanWarps ? s_cnt[lane] : 0;
                int incl = v;
#pragma unroll
                for (int o = 1; o < kPlanWarps; o <<= 1) { const int z = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += z; }
                const int before = __shfl_sync(0xffffffffu, incl - v, warp);
                msel = __shfl_sync(0xffffffffu, incl, kPlanWarps - 1);
#pragma unroll
                for (int j = 0; j < kChunks; ++j)
                    if (at[j] >= 0 && before + at[j] < kSpRound) { const int e = j * kPlanThreads + tid; r_e[before + at[j]] = e; pdone[e] = 1; }      // (beyond the cap: next round)
                msel = msel < kSpRound ? msel : kSpRound;
                __syncthreads();
            }
            if (msel == 0) {
                if (round_no == 0) round_no = 1;
                // Nothing published may beat the best score.  A block whose last bound may do so could hold more; and all of them may,
                // if bounds were left out as unlikely that it turns out may win.
                const bool unlikely = likely >= bar.lo;
                bool again = false;
                if (tid < G) {
                    const int e = (kSpTop - 1) * G + tid;
                    again = unlikely || (pidx[e] >= 0 && pkey[e] >= bar.lo);
                    s_refresh[tid] = again ? 1 : 0;
                }
                if (!__syncthreads_or(again)) break;
                if (again_published) { failed = true; break; }       // (cannot be: what is published under a floor may beat it)
                again_published = true;
                if (unlikely) likely = 0;
                if (s_refresh[c]) scan(false, true);
                if (!grid_barrier(A.bar, G, gen)) { failed = true; break; }
                barrier_since_booking = true;
                load(pbuf, true, nullptr);
                pbuf ^= 1;
                continue;
            }
            round_no += 1;
            again_published = false;
            long long sz = 0;
            ull cost = 1;
            int own = -1;                                                           // the thread's period << 1 | destination
            if (const int r = tid; r < msel) {
                const int i = own = pidx[r_e[r]], p = i >> 1, d = i & 1;
                r_ap[r] = A.geo_a[d * A.geo_stride + p]; r_bp[r] = A.geo_b[d * A.geo_stride + p];
                r_s[r] = sz = A.bytes[A.per_t[p]];
                cost = 2ull * (ull)A.geo_t[d * A.geo_stride + p];
#pragma unroll
                for (int q = 0; q < kSpLimbs; ++q) r_acc[q * kSpRound + r] = 0;
            }
            // (the largest tensor of the round, rounded up: bytes are below 2^40)
            if (const unsigned m = __reduce_max_sync(0xffffffffu, (unsigned)(sz >> 8)); lane == 0) s_fk[warp] = m;
            if (tid == 0) { s_nmid = 0; s_nedge = 0; }
            __syncthreads();
            auto add = [&](int r, u128 v) {
#pragma unroll
                for (int q = 0; q < kSpLimbs; ++q) {                                 // (a 64-bit atomic would be a compare-and-swap loop)
                    const unsigned x = (unsigned)(v >> (21 * q)) & 0x1fffffu;
                    if (x) atomicAdd(&r_acc[q * kSpRound + r], x);
                }
            };
            // benefit of local tile lt for period r, slot by slot, by one warp; every lane's share
            auto slots = [&](int r, int lt) {
                const int t0 = (lt * G + c) * kSpTile, ap = r_ap[r], bp = r_bp[r];
                const long long s = r_s[r], o = off[lt];
                u128 sum = 0;
#pragma unroll
                for (int j = 0; j < kSpTile; j += 32) {
                    const int k = t0 + j + lane;
                    if (k < ap || k > bp) continue;
                    long long e = ex[lt * kSpTile + j + lane] + o;
                    e = e > s ? s : e;
                    if (e > 0) sum += (u128)(ull)e * (u128)(ull)(A.start[k + 1] - A.start[k]);
                }
                return sum;
            };
            // Tiles above capacity by the largest tensor of the round count for their whole time for every period that covers them
            // (prefix sums); tiles within capacity count for none.  What is left is few: listed.
            const long long s_max_round = ((long long)__reduce_max_sync(0xffffffffu, lane < kPlanWarps ? s_fk[lane] : 0u) + 1) << 8;
            for (int b = warp; b * 32 < my_tiles; b += kPlanWarps) {
                const int lt = b * 32 + lane;
                const longlong2 m = lt < my_tiles ? mm[lt] : make_longlong2(0, 0);
                const bool full = lt < my_tiles && m.x >= s_max_round;
                const unsigned mid = __ballot_sync(0xffffffffu, lt < my_tiles && !full && m.y > 0);
                const ull d = full ? (ull)tsum[lt] : 0ull;
                ull incl = d;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const ull y = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += y; }
                if (lt < my_tiles) t_full[lt] = incl - d;
                if (lane == 31) s_full[b] = incl;
                int at = 0;
                if (lane == 0 && mid) at = atomicAdd(&s_nmid, __popc(mid));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(mid & ((1u << lane) - 1u));
                if (mid >> lane & 1u) t_mid[at] = (unsigned)lt;
            }
            __syncthreads();
            // a thread per period, two if there are enough (one of them for every other listed tile): whole tiles [l0, l1]; the two at
            // the ends, if they are covered in part, are listed for the warps
            const bool two = msel <= kPlanThreads / 2;
            const int nmid = s_nmid, r_me = two ? tid & (kPlanThreads / 2 - 1) : tid, half = two ? tid / (kPlanThreads / 2) : 0;
            const bool active = r_me < msel;
            long long s_me = 0;
            int l0 = 0, l1 = -1;
            u128 sum_me = 0;
            if (active) {
                const int ap = r_ap[r_me], bp = r_bp[r_me], ta = (ap + kSpTile - 1) / kSpTile, tb = bp == K - 1 ? NT - 1 : (bp + 1) / kSpTile - 1;
                s_me = r_s[r_me];
                l0 = ta > c ? (ta - c + G - 1) / G : 0; l1 = tb >= c ? (tb - c) / G : -1;
                if (half == 0) {
                    if (l0 <= l1) {
                        ull time = t_full[l1] + (mm[l1].x >= s_max_round ? (ull)tsum[l1] : 0ull) - t_full[l0];
                        for (int b = l0 / 32; b < l1 / 32; ++b) time += s_full[b];
                        sum_me = (u128)time * (u128)(ull)s_me;
                    }
                    const int ea = ap / kSpTile, eb = bp / kSpTile;
                    if (ea < ta && ea % G == c && mm[ea / G].y > 0) s_edge[atomicAdd(&s_nedge, 1)] = (unsigned)r_me << 20 | (unsigned)(ea / G);
                    if (eb > tb && (eb != ea || ea >= ta) && eb % G == c && mm[eb / G].y > 0) s_edge[atomicAdd(&s_nedge, 1)] = (unsigned)r_me << 20 | (unsigned)(eb / G);
                }
            }
            __syncthreads();
            // (the last warps first: the others sort meanwhile)
#pragma unroll 1
            for (int x = kPlanWarps - 1 - warp, nedge = s_nedge; x < nedge; x += kPlanWarps) {
                const int r = (int)(s_edge[x] >> 20);
                const u128 v = warp_sum_u128(slots(r, (int)(s_edge[x] & 0xfffffu)));
                if (lane == 0) add(r, v);
            }
            const bool direct = msel * nmid <= kSpDirect;
            if (direct) {
#pragma unroll 1
                for (int x = warp; x < msel * nmid; x += kPlanWarps) {
                    const int r = x % msel, lt = (int)t_mid[x / msel], t0 = (lt * G + c) * kSpTile;
                    if (t0 < r_ap[r] || (t0 + kSpTile - 1 > r_bp[r] && r_bp[r] != K - 1)) continue;      // (not, or in part)
                    const u128 v = warp_sum_u128(slots(r, lt));
                    if (lane == 0) add(r, v);
                }
            } else {
#pragma unroll 1
                for (int n0 = 0; n0 < nmid; n0 += kSpSort) {
                    if (n0) __syncthreads();                                        // (the sorted tiles are free)
                    if (warp < kSpSort && n0 + warp < nmid) {
                        const int lt = (int)t_mid[n0 + warp], t0 = (lt * G + c) * kSpTile, n = K - t0 < kSpTile ? K - t0 : kSpTile;
                        SpSorted &q = sorted[warp];
                        const long long o = off[lt];
                        long long v[2];
                        unsigned d[2];
                        int rank[2] = {0, 0};
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int x = h * 32 + lane;
                            d[h] = x < n ? (unsigned)(A.start[t0 + x + 1] - A.start[t0 + x]) : 0u;
                            const long long e = x < n ? ex[lt * kSpTile + x] + o : 0;
                            // (with the slot as the lowest bits: no two are equal)
                            v[h] = x < n ? (e < 0 ? 0 : e > ((long long)1 << 40) ? (long long)1 << 40 : e) << 6 | x : (long long)1 << 62;
                            q.v[x] = v[h];
                        }
                        __syncwarp();
                        const longlong2 *all = reinterpret_cast<const longlong2 *>(q.v);
#pragma unroll 4
                        for (int j = 0; j < kSpTile / 2; ++j) {                     // position of each: how many come before it
                            const longlong2 y = all[j];
#pragma unroll
                            for (int h = 0; h < 2; ++h) rank[h] += (y.x < v[h] ? 1 : 0) + (y.y < v[h] ? 1 : 0);
                        }
                        __syncwarp();
#pragma unroll
                        for (int h = 0; h < 2; ++h) if (h * 32 + lane < n) { q.v[rank[h]] = v[h] >> 6; q.d[rank[h]] = d[h]; }
                        __syncwarp();
                        // prefix sums: two consecutive entries per lane
                        const bool i0 = 2 * lane < n, i1 = 2 * lane + 1 < n;
                        const ull v0 = i0 ? (ull)q.v[2 * lane] : 0ull, v1 = i1 ? (ull)q.v[2 * lane + 1] : 0ull;
                        const unsigned d0 = i0 ? q.d[2 * lane] : 0u, d1 = i1 ? q.d[2 * lane + 1] : 0u;
                        const ull a0 = (v0 & 0xfffffull) * d0, a1 = (v1 & 0xfffffull) * d1, b0 = (v0 >> 20) * d0, b1 = (v1 >> 20) * d1;
                        unsigned sd = d0 + d1;
                        ull sa = a0 + a1, sb = b0 + b1;
#pragma unroll
                        for (int o2 = 1; o2 < 32; o2 <<= 1) {
                            const unsigned yd = __shfl_up_sync(0xffffffffu, sd, o2);
                            const ull ya = __shfl_up_sync(0xffffffffu, sa, o2), yb = __shfl_up_sync(0xffffffffu, sb, o2);
                            if (lane >= o2) { sd += yd; sa += ya; sb += yb; }
                        }
                        __syncwarp();
                        q.d[2 * lane] = sd - d1 - d0; q.lo[2 * lane] = sa - a1 - a0; q.hi[2 * lane] = sb - b1 - b0;
                        q.d[2 * lane + 1] = sd - d1; q.lo[2 * lane + 1] = sa - a1; q.hi[2 * lane + 1] = sb - b1;
                        if (lane == 31) { q.d[kSpTile] = sd; q.lo[kSpTile] = sa; q.hi[kSpTile] = sb; }
                        if (lane == 0) { q.n = n; q.lt = lt; }
                    }
                    __syncthreads();
                    if (active) {
                        const int more = nmid - n0 < kSpSort ? nmid - n0 : kSpSort;
#pragma unroll 1
                        for (int m = half; m < more; m += two ? 2 : 1) {
                            const SpSorted &q = sorted[m];
                            if (q.lt < l0 || q.lt > l1) continue;
                            int j = 0;                                              // slots less than s above capacity
#pragma unroll
                            for (int h = kSpTile / 2; h > 0; h >>= 1)
                                if (j + h <= q.n && q.v[j + h - 1] < s_me) j += h;
                            if (j < q.n && q.v[j] < s_me) ++j;
                            sum_me += ((u128)q.hi[j] << 20) + (u128)q.lo[j] + (u128)(ull)s_me * (u128)(ull)(q.d[kSpTile] - q.d[j]);
                        }
                    }
                }
            }
            if (half != 0 && sum_me != 0) add(r_me, sum_me);
            __syncthreads();
            // this block's shares go into the grid-wide sums: the low 44 bits and the rest on their own, so that neither needs a carry
            // and no block waits for an answer
            if (half == 0 && active) {
                const int r = r_me;
                u128 v = sum_me;
#pragma unroll
                for (int q = 0; q < kSpLimbs; ++q) v += (u128)r_acc[q * kSpRound + r] << (21 * q);
                ull *dst = S.partials + (size_t)pp * 2 * kSpRound + r;
                const ull lo = (ull)v & 0xfffffffffffull, hi = (ull)(v >> 44);
                if (lo) asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(dst), "l"(lo) : "memory");
                if (hi) asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(dst + kSpRound), "l"(hi) : "memory");
            }
            if (!grid_barrier(A.bar, G, gen)) { failed = true; break; }
            barrier_since_booking = true;
            // (the buffer used two rounds from now was last read one round ago: block 0 clears it)
            if (c == 0) for (int j = tid; j < kSpRound * 2; j += kPlanThreads) S.partials[(size_t)((pp + 2) % 3) * kSpRound * 2 + j] = 0;
            Cand x;
            x.ben = 0; x.cost = 1; x.idx = -1; x.dest = -1;
            unsigned key = 0;
            if (tid < msel) {
                const int i = own, p = i >> 1;
                const ull *src = S.partials + (size_t)pp * 2 * kSpRound + tid;
                const u128 tot = ((u128)__ldcg(src + kSpRound) << 44) + __ldcg(src);
                x.ben = tot; x.cost = cost; x.idx = tot == 0 ? -1 : p; x.dest = i & 1;
                key = sp_key(tot, x.cost);
                const int e = owner_entry(p);
                if (e >= 0) {
                    S.c_ben_lo[p] = (ull)tot; S.c_ben_hi[p] = (ull)(tot >> 64);
                    uint4 q = hot[e];
                    q.x = key; q.w |= kSpFresh;
                    hot[e] = q;
                }
            }
            const Cand b = best_of(x, key);
            if (cand_beats(b, gBest)) gBest = b;
            pp = (pp + 1) % 3;
            __syncthreads();
        }
        if (failed) { status = -2; break; }
        // The bookings have to be there before the next pass.  And where the last choice compared other blocks' periods exactly, by the
        // benefits and costs in global memory, nobody may restart a period (begin_period in the next pass) before all blocks have
        // read them: a block that comes late would choose otherwise than the rest.  (`compared` is the same in all blocks: they see
        // the same bounds and the same best score.  Rare, and a barrier is a tenth of an iteration.)
        if (!barrier_since_booking || compared) { if (!grid_barrier(A.bar, G, gen)) { status = -2; break; } }
        // ---------------- D: decide
        if (gBest.idx < 0) { status = G10_EXHAUSTED; break; }
        {
            const int p = gBest.idx, X = gBest.dest;
            w.idx = p; w.dest = X; w.a = A.per_u[p] + 1; w.b = A.per_v[p] - 1;
            w.ap = A.geo_a[X * A.geo_stride + p]; w.bp = A.geo_b[X * A.geo_stride + p]; w.t = A.geo_t[X * A.geo_stride + p];
            w.s = A.bytes[A.per_t[p]];
            w.t_r = A.start[w.a]; w.t_end = A.start[w.b + 1];
            last_key = (float)cand_key(gBest);
            float least = last_key;
#pragma unroll
            for (int j = kSpPast - 1; j > 0; --j) { won[j] = won[j - 1]; least = fminf(least, won[j]); }
            won[0] = last_key;
            likely = __float_as_uint(least * kLikely);
            if (X == G10_DEST_SSD) bytes_ssd += w.s; else bytes_host += w.s;
        }
        n_mig += 1;
        pending = true;
    }
    __syncthreads();
    for (int x = tid; x < my_tiles * kSpTile; x += kPlanThreads) {
        const int64_t k = ((int64_t)(x / kSpTile) * G + c) * kSpTile + x % kSpTile;
        if (k < K) A.P[k] = ex[x] + off[x / kSpTile] + A.cap;
    }
    if (c == 0 && tid == 0) *S.done = 1u;
    {
        // the peak of what is left (every block's own, then all of them)
        long long m = 0;
        for (int x = tid; x < my_tiles; x += kPlanThreads) m = mm[x].y + A.cap > m ? mm[x].y + A.cap : m;
        m = block_max_i64(m, s_max);
        if (tid == 0) A.peak_part[c] = m;
    }
    if (status != -2 && !grid_barrier(A.bar, G, gen)) status = -2;
    if (status != -2) {
        long long m = 0;
        for (int j = tid; j < G; j += kPlanThreads) { const long long x = __ldcg(&A.peak_part[j]); m = x > m ? x : m; }
        peak = block_max_i64(m, s_max);
    }
    plan_epilogue(A, c, G, gen, status, peak, n_mig, rounds, bytes_ssd, bytes_host);
}

// Shared memory a launch can offer (0 if a query fails).
static int spread_budget()
{
    static int known[kMaxDevices];
    return dynamic_smem_room((const void *)k_plan_spread, known);
}

// Worth launching: the timeline leaves room for at least some periods (their number is counted on the device, which decides).
bool plan_spread_possible(int64_t K, int64_t E)
{
    const int G = current_sm_count(), budget = spread_budget();
    return G > 0 && G <= kLazyMaxBlocks && G <= kPlanThreads && K >= 1 && K <= kSpMaxSlots && E >= 1 && budget > 0 && spread_layout(K, E < 4096 ? E : 4096, G).total <= (size_t)budget;
}

cudaError_t launch_plan_spread(const PlanArgs &A_in, const Workspace &w, cudaStream_t s)
{
    PlanArgs A = A_in;
    A.bar = (GridBarrier *)(w.barrier2);
    SpreadArgs S;
    S.c_ben_lo = w.c_ben_lo; S.c_ben_hi = w.c_ben_hi; S.c_cost = w.c_cost; S.props = (SpProp *)w.lazy_props; S.partials = w.lazy_partials;
    S.flag = w.spread_flag; S.done = w.one_done; S.smem_bytes = spread_budget();
    void *args[] = {&A, &S};
    if (const cudaError_t e = allow_launch((const void *)k_plan_spread, (size_t)S.smem_bytes, 1); e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel((const void *)k_plan_spread, dim3(current_sm_count()), dim3(kPlanThreads), args, (size_t)S.smem_bytes, s);
}

#ifdef G10_TEST_HOOKS
// What the tests want to know of the layout: offsets of the arrays in the order of the struct, then the total.
extern "C" int32_t g10_test_spread_layout(int64_t K, int64_t Pn, int32_t G, int64_t *out /* [18] */)
{
    const SpreadLayout l = spread_layout(K, Pn, G);
    const size_t v[] = {l.mm, l.hot, l.r_acc, l.r_s, l.r_e, l.r_ap, l.r_bp, l.edge, l.sorted, l.mid, l.full, l.pkey, l.pidx, l.pdone, l.ex, l.off, l.tsum, l.total};
    for (int j = 0; j < 18; ++j) out[j] = (int64_t)v[j];
    return (int32_t)sizeof(SpSorted);
}
extern "C" int32_t g10_test_spread_budget(void) { return spread_budget(); }
#endif

}  // namespace g10
