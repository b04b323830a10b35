// Core-first match enumeration over the compact path index (Section III.B,
// step 2) with the literal check and violation output (Section II) fused into
// the last level.
//
// Execution model: a breadth-first / depth-first hybrid over many GFD slots at
// once. Each slot keeps one buffer of partial matches per level. A step takes
// a bounded chunk of "work items" from the deepest unfinished level of every
// active slot: work item w of level l is the pair (partial match r, o-th index
// edge of r's tree parent), found by binary search in the exclusive prefix of
// the rows' fan-outs, so hub vertices are split evenly over threads. Each work
// item yields at most one partial match of level l+1, so a level-l chunk of
// `cap` items always fits the next buffer (steps that make the second-to-last
// level take more, since they store few of theirs; see control_step); when a level is
// exhausted the slot pops back to the previous level (depth-first), bounding memory.
//
// A candidate v for pattern node u = order[i] extending partial match m passes
// when: v != m[q] for earlier label-compatible levels q (injectivity), and for
// every earlier level q and both directions, the data-graph edge between v and
// m[q] agrees with the pattern (present with an equal label where Q has the
// edge, absent where it has not: a match may not contain additional edges,
// Section II; the CFL-Match index alone would allow them, Section III). The
// spanning-tree edge to the parent is guaranteed by the index and skipped.
//
// Survivors are appended with one atomic per warp on a packed 64-bit counter
// (rows << 40 | fan-out sum), which gives each row both its index and the
// exclusive prefix of fan-outs needed by the next step's search, consistently.
//
// The scheduler (k_control) runs in one block between steps. Two drivers: a
// persistent cooperative kernel with a bounded grid barrier between phases, or
// a host loop of (expand, control) launches, optionally captured in CUDA graphs.
#include <cub/cub.cuh>

#include <algorithm>
#include <type_traits>

#include "engine.h"

namespace gfd {

namespace {

constexpr int CTRL_THREADS = 1024;
constexpr uint64_t LAST_LEVEL_CHUNK = 1ull << 25;  // most work items per step at the last two levels
// Last-level items that a step of the level before should lead to at most, all its
// slots together, and that it may expand in place for want of a row (0.3 s for lists
// of 200,000, far below the limit of a wait at the grid barrier).
constexpr uint64_t FUSED_STEP_WORK = 1ull << 33;
// Longest candidate list expanded in place for want of a row: one warp's work, up to
// a tile of them (2^27 items, about a second) before it looks for the next.
constexpr uint32_t SPILL_FANOUT = 1u << 18;
// A warp counts a tile's matches, at most SPILL_FANOUT of each item, in 32 bits.
static_assert(32ull * MAX_TILE_ITERS * SPILL_FANOUT < 1ull << 32, "matches of a tile");
// generator stored in a row for a next level that starts a pattern component:
// its candidates are the level's candidate list (fan-out |C| for every row)
constexpr int GEN_LIST = 4;

__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Per-thread counters of the counting pass (empty unless COUNT), added into
// Sched::cnt once per warp at the end of the expansion.
template <bool COUNT>
struct Counters {
    __device__ __forceinline__ void add(int, uint64_t) {}
    __device__ __forceinline__ uint32_t* loads() { return nullptr; }
    __device__ __forceinline__ void iteration(bool) {}
    __device__ __forceinline__ void mark() {}
    __device__ __forceinline__ void cycles(int) {}
    __device__ __forceinline__ void flush(Sched*) {}
};
template <>
struct Counters<true> {
    uint64_t c[N_CNT] = {};
    uint32_t search_loads = 0;  // of the current warp iteration
    __device__ __forceinline__ void add(int i, uint64_t v) { c[i] += v; }
    __device__ __forceinline__ uint32_t* loads() { return &search_loads; }
    long long t0 = 0;  // clock at the start of the current phase
    __device__ __forceinline__ void mark() { t0 = clock64(); }
    // SM cycles since mark() into counter i (lane 0 counts for the warp)
    __device__ __forceinline__ void cycles(int i) {
        const long long t = clock64();
        if ((threadIdx.x & 31) == 0) c[i] += (uint64_t)(t - t0);
        t0 = t;
    }
    // end of a warp iteration (all lanes): the slowest lane's search loads
    __device__ __forceinline__ void iteration(bool last) {
        const uint32_t mx = __reduce_max_sync(0xffffffffu, search_loads);
        if ((threadIdx.x & 31) == 0) {
            c[CNT_ITERS] += 1;
            c[CNT_ITER_MAX_LOADS] += mx;
            if (!last) c[CNT_ITERS_MID] += 1;
        }
        c[CNT_SEARCH_LOADS] += search_loads;
        search_loads = 0;
        cycles(last ? CNT_CYC_LAST : CNT_CYC_MID);
    }
    __device__ void flush(Sched* s) {
        for (int i = 0; i < N_CNT; i++) {
            uint64_t v = c[i];
            for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
            if ((threadIdx.x & 31) == 0 && v) atomicAdd((unsigned long long*)&s->cnt[i], (unsigned long long)v);
        }
    }
};

__device__ __forceinline__ uint32_t ceil_log2_1(uint32_t d) { return 32 - __clz(d); }  // ceil(log2(d + 1))

// Label of the data-graph edge a -> b, or NOEDGE: binary search in the shorter
// of out(a) and in(b) (both sorted by neighbour id). loads (counting pass
// only, else null) accumulates the adjacency entries read.
__device__ __forceinline__ int32_t edge_label(const DevGraph& g, uint32_t a, uint32_t a_out0, uint32_t a_out1,
                                              uint32_t b, uint32_t b_in0, uint32_t b_in1,
                                              uint32_t* loads = nullptr) {
    const uint32_t* arr;
    uint32_t lo, hi, key;
    if (a_out1 - a_out0 <= b_in1 - b_in0) {
        arr = g.out_adj;
        lo = a_out0;
        hi = a_out1;
        key = b;
    } else {
        arr = g.in_adj;
        lo = b_in0;
        hi = b_in1;
        key = a;
    }
    const uint32_t end = hi;
    const uint32_t kk = key << g.lbits;
    #pragma unroll 1
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (loads) ++*loads;
        if (__ldg(arr + mid) < kk) lo = mid + 1;
        else hi = mid;
    }
    if (lo < end) {
        if (loads) ++*loads;
        const uint32_t p = __ldg(arr + lo);
        if ((p >> g.lbits) == key) return (int32_t)(p & g.lmask);
    }
    return NOEDGE;
}

// A partial match is a column in shared memory: level q at m[32 q]. Vertex of
// level q when that of level lv is given in a register (v) and the column holds
// the earlier ones.
__device__ __forceinline__ uint32_t level_vertex(const uint32_t* m, int q, int lv, uint32_t v) {
    return q == lv ? v : m[q << 5];
}
__device__ __forceinline__ bool lit_holds_at(const DevGraph& g, const DevLit& L, const uint32_t* m, int lv, uint32_t v,
                                             uint32_t* reads = nullptr) {
    if (reads) ++*reads;
    const int32_t va = __ldg(g.attrs + (uint64_t)L.a * g.n + level_vertex(m, L.xl, lv, v));
    if (va == GFD_ATTR_ABSENT) return false;
    if (L.kind == 0) return va == L.c;
    if (reads) ++*reads;
    const int32_t vb = __ldg(g.attrs + (uint64_t)L.b * g.n + level_vertex(m, L.yl, lv, v));
    return vb != GFD_ATTR_ABSENT && va == vb;
}

// Partial matches of the second-to-last level with at most this many
// candidates at the last level are expanded by the warp that makes them,
// without being stored.
constexpr uint32_t FUSE_FANOUT = 64;
static_assert(FUSE_FANOUT <= SPILL_FANOUT);
// Tiles of a step that fuses the last level are this many times smaller.
constexpr uint64_t FUSED_TILE_DIV = 4;
// Number the last level's tiles after the other intermediate levels' (else
// both are numbered together, in slot order).
constexpr bool LAST_LEVEL_TILES_LAST = true;

// Loads of data rewritten between steps (frontier rows and prefixes, the
// per-step tile prefix): plain weak loads, which may be served from L1. In the
// persistent kernel the grid barrier orders them after the previous step's
// writes: every writer's block fences at gpu scope before arriving, each
// block's thread 0 fences at gpu scope after observing the release, and the
// block barrier orders the block's other threads after that fence, so by the
// PTX memory model the loads observe the writes (the pattern of a cooperative
// grid synchronisation). In the host-driven loop the kernel boundary orders them.
__device__ __forceinline__ uint32_t ld_front(const uint32_t* p) { return *p; }
__device__ __forceinline__ uint64_t ld_front(const uint64_t* p) { return *p; }

// r in [lo, hi) with S[r] <= w < S[r+1]: the search limited to the rows of a tile.
__device__ __forceinline__ uint32_t find_row_in(const uint32_t* S, uint32_t lo, uint32_t hi, uint64_t w) {
    #pragma unroll 1
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if ((uint64_t)__ldg(S + mid) <= w) lo = mid;
        else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ uint32_t find_row_in(const uint64_t* S, uint32_t lo, uint32_t hi, uint64_t w) {
    #pragma unroll 1
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldcg((const unsigned long long*)S + mid) <= w) lo = mid;
        else hi = mid;
    }
    return lo;
}

// One half of a vertex's neighbourhood signature: 0 its out-neighbours, 1 its
// in-neighbours. An edge a -> b needs both b's bit in a's out-signature and
// a's bit in b's in-signature, so either clear bit proves it absent.
__device__ __forceinline__ uint64_t sig_half(const DevGraph& g, uint32_t x, int half) {
    return __ldg(reinterpret_cast<const unsigned long long*>(g.sig) + 2 * (uint64_t)x + half);
}

// May v be in the adjacency row [e0, e0 + d) of x (in: its in-neighbours)?
__device__ __forceinline__ bool row_filter(const DevGraph& g, bool in, uint32_t e0, uint32_t d, uint32_t v) {
    const uint32_t bit = filter_bit(v, d);
    return (__ldg((in ? g.in_filter : g.out_filter) + e0 + (bit >> 3)) >> (bit & 7)) & 1u;
}

// position of v in the sorted candidate list of a level: O(1) from the bitmap
// and its per-word popcount prefix
__device__ __forceinline__ int32_t cand_rank(const uint32_t* bm, const uint32_t* rank, uint32_t v) {
    return (int32_t)(__ldg(rank + (v >> 5)) + __popc(__ldg(bm + (v >> 5)) & ((1u << (v & 31)) - 1u)));
}

// Warp-parallel search: largest r in [lo, hi) with S[r] <= w, given S[lo] <= w.
// Each round probes 32 evenly spaced entries and keeps the last one <= w.
template <typename T>
__device__ __forceinline__ uint32_t warp_find(const T* S, uint64_t lo, uint64_t hi, uint64_t w, int lane) {
    #pragma unroll 1
    while (hi - lo > 32) {
        const uint64_t step = (hi - lo + 31) / 32;
        const uint64_t idx = lo + (uint64_t)lane * step;
        const bool le = idx < hi && (uint64_t)ld_front(S + idx) <= w;
        const uint32_t b = __ballot_sync(0xffffffffu, le);
        const int j = 31 - __clz(b);
        lo = lo + (uint64_t)j * step;
        hi = min(hi, lo + step);
    }
    const uint64_t idx = lo + lane;
    const bool le = idx < hi && (uint64_t)ld_front(S + idx) <= w;
    const uint32_t b = __ballot_sync(0xffffffffu, le);
    return (uint32_t)(lo + 31 - __clz(b));
}

// Exclusive warp scan of 64-bit values; *total receives the warp's sum.
__device__ __forceinline__ uint64_t warp_excl_scan(uint64_t x, int lane, uint64_t* total) {
    uint64_t incl = x;
    #pragma unroll 1
    for (int d = 1; d < 32; d <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    *total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - x;
}

// A row filter: bits of it from base on (0: no filter to pass).
struct FilterRow {
    const uint8_t* base;
    uint32_t bits;
    __device__ __forceinline__ bool may_hold(uint32_t v) const {
        const uint32_t b = filter_bit_of(v, bits);
        return (__ldg(base + (b >> 3)) >> (b & 7)) & 1u;
    }
};

// Fused expansion: the last-level candidates of one partial match in the warp's
// sequence, and the row filter they are looked up in. src: where they start in their
// generator's source - where they start in the sequence.
struct LastList {
    const uint8_t* base;
    uint32_t bits;
    uint32_t src;
};

constexpr int LAST_WINDOWS = 2;  // windows of 32 candidates in flight at the last level

// Per warp in (dynamic) shared memory.
struct WarpShared {
    uint32_t chk[2 * MAXK];   // the current tile's pair checks, packed
    uint32_t chk2[2 * MAXK];  // the last level's, for fused expansion
    LastList list[32];        // fused expansion: the partial matches' candidates, in order
    uint8_t who[32];          // whose each is: lane | generator << 5
    int32_t* rows;            // where the tile's new partial matches go
    uint64_t* wpre;
    uint64_t cap;
    uint32_t qv[32 + 32 * LAST_WINDOWS];  // last-level candidates waiting for their other checks,
    uint8_t qo[32 + 32 * LAST_WINDOWS];   // and whose they are: lane | generator << 5
    __device__ uint32_t* m(int col) { return reinterpret_cast<uint32_t*>(this + 1) + col; }  // [32 q + col]: the columns
};
// columns for patterns of up to kmax nodes (rows are loaded in groups of four)
__host__ __device__ constexpr int column_words(int kmax) { return ((kmax + 3) & ~3) * 32; }
constexpr size_t warp_shared_bytes(int kmax) { return sizeof(WarpShared) + 4 * (size_t)column_words(kmax); }

// Every pattern pair of v, the candidate of a level, with the earlier images in
// the column m, but check `skip`: the n packed checks cw, the first nreq of them
// required edges. v's signature comes first (one load for all pairs): a clear bit
// settles an absent edge and refutes a required one. Only the pairs it leaves
// open look into the other end's row filter, and only those that leaves open
// search the shorter adjacency list.
template <bool COUNT>
__device__ __forceinline__ bool pairs_agree(const DevGraph& g, const uint32_t* m, const uint32_t* cw, int n, int nreq,
                                            int skip, uint32_t v, uint32_t& probes, Counters<COUNT>& cn) {
    if (n == 0) return true;
    const ulonglong2 sv = __ldg(g.sig + v);  // out-, in-neighbours
    cn.add(CNT_SIG_LOADS, 1);
    uint32_t open = 0;
    #pragma unroll 1
    for (int c = 0; c < n; c++) {
        const uint32_t wd = cw[c];
        const uint32_t x = m[(wd & 15u) << 5];
        const uint64_t half = (wd >> 4) & 1u ? sv.x : sv.y;  // edge v -> x, else x -> v
        open |= (uint32_t)((half >> sig_bit(x)) & 1ull) << c;
    }
    // All pairs are tested here. Of those the signature leaves open, the counting pass
    // takes back the ones not looked up any more (doing so in every run, for the
    // statistic, cost 2 % of the large batch's enumeration).
    probes += n - (skip >= 0);
    cn.add(CNT_CHECKS, n - (skip >= 0));
    // counting pass: absent edges, in order up to the first that is there (check c; n: none)
    auto count_absent = [&](int c1) {
        for (int c = nreq; COUNT && c < min(c1 + 1, n); c++) {
            const uint32_t x = m[(cw[c] & 15u) << 5];
            const bool out = (cw[c] >> 4) & 1u;
            const uint32_t dv = out ? g.out_off[v + 1] - g.out_off[v] : g.in_off[v + 1] - g.in_off[v];
            const uint32_t dx = out ? g.in_off[x + 1] - g.in_off[x] : g.out_off[x + 1] - g.out_off[x];
            cn.add(CNT_NEG_CHECKS, 1);
            cn.add(CNT_NEG_LOGD, ceil_log2_1(min(dv, dx)));
        }
    };
    uint32_t required = (1u << nreq) - 1u;  // (at most 2 (MAXK - 1) = 30 checks)
    if (skip >= 0) {
        open &= ~(1u << skip);
        required &= ~(1u << skip);
    }
    if (COUNT) cn.add(CNT_SIG_SETTLED, n - (skip >= 0) - __popc(open));
    if ((open & required) != required) {
        cn.add(CNT_CHECKS, -(uint64_t)__popc(open));
        return false;
    }
    #pragma unroll 1
    for (; open; open &= open - 1) {
        const int c = __ffs(open) - 1;
        const uint32_t wd = cw[c];
        const uint32_t x = m[(wd & 15u) << 5];
        const bool out = (wd >> 4) & 1u;
        const int32_t ex = (int32_t)(int16_t)(wd >> 16);
        int32_t gl = NOEDGE;
        cn.add(CNT_SIG_LOADS, 1);
        const uint32_t* const off = out ? g.in_off : g.out_off;
        const uint32_t e0 = __ldg(off + x), e1 = __ldg(off + x + 1);
        if (e0 < e1 && row_filter(g, out, e0, e1 - e0, v)) {
            cn.add(CNT_SEARCHES, 1);
            gl = out ? edge_label(g, v, g.out_off[v], g.out_off[v + 1], x, e0, e1, cn.loads())
                     : edge_label(g, x, e0, e1, v, g.in_off[v], g.in_off[v + 1], cn.loads());
        } else {
            cn.add(CNT_SIG_SETTLED, 1);
        }
        if (!exp_ok(ex, gl)) {
            cn.add(CNT_CHECKS, 1 - (uint64_t)__popc(open));
            count_absent(c);
            return false;
        }
    }
    count_absent(n);
    return true;
}

// Does the spanning-tree edge between v and its parent's image xp agree? (v comes
// from another generator than the parent's index edges.)
template <bool COUNT>
__device__ __forceinline__ bool tree_edge_agrees(const DevGraph& g, const LevelPlan& P, uint32_t xp, uint32_t v,
                                                 uint32_t& probes, Counters<COUNT>& cn) {
    // the parent's signature first, then v's
    bool maybe = (sig_half(g, xp, P.tdir ? 0 : 1) >> sig_bit(v)) & 1ull;
    cn.add(CNT_SIG_LOADS, 1);
    if (maybe) {
        maybe = (sig_half(g, v, P.tdir ? 1 : 0) >> sig_bit(xp)) & 1ull;
        cn.add(CNT_SIG_LOADS, 1);
    }
    int32_t gl = NOEDGE;
    cn.add(CNT_CHECKS, 1);
    if (maybe) {
        cn.add(CNT_SEARCHES, 1);
        gl = P.tdir ? edge_label(g, xp, g.out_off[xp], g.out_off[xp + 1], v, g.in_off[v], g.in_off[v + 1], cn.loads())
                    : edge_label(g, v, g.out_off[v], g.out_off[v + 1], xp, g.in_off[xp], g.in_off[xp + 1], cn.loads());
    } else {
        cn.add(CNT_SIG_SETTLED, 1);
    }
    probes++;
    return exp_ok(P.tlab, gl);
}

// Where a last-level candidate (plan P, checks cw, from generator gen) of the
// partial match in column m must be found first: the row filter of the first
// required edge that is not the generator's, at its image. bits 0: none.
__device__ __forceinline__ FilterRow first_row(const DevGraph& g, const LevelPlan& P, const uint32_t* m,
                                               const uint32_t* cw, int gen) {
    FilterRow f{nullptr, 0};
    const int c = gen >= 1 && gen != GEN_LIST && P.gen[gen - 1] == 0 ? 1 : 0;
    if (c < P.nreq) {
        const uint32_t x = m[(cw[c] & 15u) << 5];
        const bool in = (cw[c] >> 4) & 1u;  // edge v -> x: v among x's in-neighbours
        const uint32_t* const off = in ? g.in_off : g.out_off;
        const uint32_t e0 = __ldg(off + x);
        f.base = (in ? g.in_filter : g.out_filter) + e0;
        f.bits = filter_bits(__ldg(off + x + 1) - e0);
        // (a generator's list is no longer than this one, so it is not empty)
    }
    return f;
}

// The loops below have few rounds and are not unrolled (left to itself the
// compiler unrolls most of them by four): the expansion's code, 150 KB unrolled and
// 119 KB like this, does not fit the instruction caches, and its warps are each in
// another part of it. Batch of 256 GFDs on 4M vertices: 144 -> 135 ms, a session of
// 48 requests 39 -> 36 ms of rounds.
//
// The expansion step, warp-synchronous: every warp takes its own tiles of
// work items (no block-wide barrier in the loop). A tile belongs to one slot
// and one level; the warp finds them (and the rows the tile covers) with
// lane-parallel searches, then processes 32 work items per iteration.
// GEN = false: the common case (connected patterns, X checked at the last
// level only), compiled without the general paths so that it keeps its
// registers; GEN = true adds component starts and X pushed down.
//
// The last level has most of the work items, and most fail their first required
// edge. So its candidates pass two stages: every lane fetches two and looks them up
// in the row filter of that edge's other end (FilterRow, set up once per partial
// match); those that pass wait in a queue until 32 are together for the other
// checks, the literals and the output, which then run with full warps.
template <int NT, bool GEN, bool COUNT>
__device__ void expand_warps(const EnumArgs& A) {
    extern __shared__ __align__(16) uint8_t s_dyn[];
    WarpShared& W = *reinterpret_cast<WarpShared*>(s_dyn + (threadIdx.x >> 5) * (sizeof(WarpShared) + 4u * A.columns));
    Counters<COUNT> cn;
    uint32_t attr_reads = 0;
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    uint32_t* const m = W.m(lane);
    uint32_t* const cw = W.chk;
    uint32_t* const cw2 = W.chk2;
    const uint64_t gwarp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const DevGraph& g = A.g;
    const uint32_t total_tiles = *(volatile uint32_t*)&A.sched->total_tiles;
    uint32_t probes = 0;  // a statistic
    #pragma unroll 1
    for (uint64_t t = gwarp; t < total_tiles;) {
        cn.mark();
        // the step's tiles: those of fusing slots first, then those of the other
        // intermediate levels, then the last level's
        const uint32_t* tb = A.tile_base;
        if (t >= __ldcg(A.tile_base + A.n_slots)) tb += A.n_slots + 1;
        if (t >= __ldcg(A.tile_base + 2 * A.n_slots + 1)) tb = A.tile_base + 2 * (A.n_slots + 1);
        const int s = (int)warp_find(tb, 0, (uint64_t)A.n_slots, t, lane);
        const SlotDesc* __restrict__ D = A.slots + s;
        SlotState* S = A.state + s;
        const int k = D->k;
        // scheduler fields are rewritten between steps: read them through L2
        const int l = __ldcg(&S->cur);
        const int i = k == 1 ? 0 : l + 1;  // level being matched
        const bool last = i == k - 1;
        const uint64_t tile = __ldcg(&S->tile);  // work items per tile of this slot in this step
        const uint64_t wb = __ldcg((const unsigned long long*)&S->cb) + (t - __ldcg(tb + s)) * tile;
        const uint64_t we = min(wb + tile, (uint64_t)__ldcg((const unsigned long long*)&S->ce));
        const LevelPlan& LP = D->lv[i];
        const int nchk = LP.nchk;
        __syncwarp();  // the previous tile's checks are no longer read
        if (lane < nchk) cw[lane] = LP.chk_w[lane];
        if (lane == 0 && !last) {
            W.rows = (int32_t*)__ldcg((const unsigned long long*)&S->rows[i]);
            W.wpre = (uint64_t*)__ldcg((const unsigned long long*)&S->wpre[i]);
            W.cap = __ldcg((const unsigned long long*)&S->cap[i]);
        }
        __syncwarp();
        const uint32_t* S0 = i > 0 ? D->cpi_off[i] : nullptr;
        const uint64_t* Sl = l >= 1 ? (const uint64_t*)__ldcg((const unsigned long long*)&S->wpre[l]) : nullptr;
        const int32_t* rows_l = l >= 1 ? (const int32_t*)__ldcg((const unsigned long long*)&S->rows[l]) : nullptr;
        const uint64_t nrows = k == 1 ? 0 : (l == 0 ? (uint64_t)S->ncand[0]
                                                    : (uint64_t)__ldcg((const unsigned long long*)&S->nrows[l]));
        const int rw = row_width(l);  // ints per row at level l: ids, positions, generator, index base
        // level 1 starts a component: root r's items are [r c1, (r+1) c1)
        const bool list1 = GEN && k > 1 && l == 0 && LP.par < 0;
        const uint64_t c1 = list1 ? (uint64_t)S->ncand[1] : 0;
        uint32_t rlo = 0, rhi1 = 0;
        if (k > 1 && !list1) {
            if (l == 0) {
                rlo = warp_find(S0, 0, nrows, wb, lane);
                rhi1 = warp_find(S0, rlo, nrows, we - 1, lane) + 1;
            } else {
                // stored rows all have fan-out >= 1, so the window search never
                // runs past the tile's last row: the end of the row range need
                // not be searched
                rlo = warp_find(Sl, 0, nrows, wb, lane);
                rhi1 = (uint32_t)nrows;
            }
        }
        uint32_t tile_matches = 0;  // (of the whole tile: below 2^32, see SPILL_FANOUT)
        // Complete matches (ok lanes: v at the last level L, the earlier levels in
        // column c): check the X literals of this level, count (with X pushed down
        // only if they hold), check Y, emit violations.
        auto finish = [&](bool ok, int L, uint32_t v, const uint32_t* c) {
            bool viol = false;
            if (ok) {
                bool x_ok = true;
                #pragma unroll 1
                for (int q = 0; q < D->nx && x_ok; q++)
                    if (!GEN || D->lit[q].lvl == L)
                        x_ok = lit_holds_at(g, D->lit[q], c, L, v, COUNT ? &attr_reads : nullptr);
                if (GEN) tile_matches += x_ok || !D->push_x;
                else tile_matches++;
                if (x_ok) {
                    bool y_ok = !D->y_false;
                    #pragma unroll 1
                    for (int q = 0; q < D->ny && y_ok; q++)
                        y_ok = lit_holds_at(g, D->lit[D->nx + q], c, L, v, COUNT ? &attr_reads : nullptr);
                    viol = !y_ok;
                }
            }
            const uint32_t vb = __ballot_sync(0xffffffffu, viol);
            if (!vb) return;
            unsigned long long base = 0;
            if (lane == 0) {
                const unsigned long long nv = __popc(vb);
                const unsigned long long old = atomicAdd((unsigned long long*)&S->n_viol, nv);
                base = D->viol ? old : atomicAdd((unsigned long long*)&A.sched->varena_used, nv);
            }
            base = __shfl_sync(0xffffffffu, base, 0);
            if (viol) {
                const uint64_t idx = base + __popc(vb & below);
                if (D->viol) {
                    // the slot's own buffer: tuples in pattern-node order
                    if (idx < D->viol_cap) {
                        int32_t* out = D->viol + idx * k;
                        #pragma unroll 1
                        for (int q = 0; q < k; q++) out[D->order[q]] = (int32_t)__ldg(g.orig + level_vertex(c, q, L, v));
                    }
                } else if (idx < A.sched->varena_cap) {
                    // the run's arena: [slot, tuple in pattern-node order]
                    int32_t* rec = A.sched->varena + idx * A.sched->vstride;
                    rec[0] = s;
                    #pragma unroll 1
                    for (int q = 0; q < k; q++) rec[1 + D->order[q]] = (int32_t)__ldg(g.orig + level_vertex(c, q, L, v));
                }
            }
        };
        // First stage of the last level (plan P, level L): an item's candidate from
        // the source of its generator,
        auto last_raw = [&](const LevelPlan& P, const uint32_t* ids, uint32_t e, int gen) -> uint32_t {
            if (gen == 0) return __ldg(ids + e);  // (index edges of the last level: ids alone)
            if (GEN && gen == GEN_LIST) return (uint32_t)__ldg(ids + e);
            return P.chk_dir[P.gen[gen - 1]] ? __ldg(g.in_adj + e) : __ldg(g.out_adj + e);
        };
        // and appending it to the queue if its row filter lets it pass.
        auto first_stage = [&](const LevelPlan& P, int L, uint32_t queued, bool ok, uint32_t raw, int who,
                               const FilterRow f) -> uint32_t {
            uint32_t v = raw;
            if (ok) {
                cn.add(CNT_ITEMS, 1);
                cn.add(CNT_ITEMS_LAST, 1);
                const int gen = who >> 5;
                const bool adjacent = gen != 0 && !(GEN && gen == GEN_LIST);
                if (adjacent) v = raw >> g.lbits;
                if (f.bits) {
                    ok = f.may_hold(v);
                    probes += !ok;
                    cn.add(CNT_SIG_LOADS, 1);
                    cn.add(CNT_CHECKS, !ok);
                    cn.add(CNT_SIG_SETTLED, !ok);
                }
                if (adjacent && ok)  // from the adjacency of the other end of a required back edge
                    ok = exp_ok(P.chk_exp[P.gen[gen - 1]], (int32_t)(raw & g.lmask)) &&
                         ((__ldg(D->bm[L] + (v >> 5)) >> (v & 31)) & 1u);
            }
            const uint32_t pass = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                const uint32_t at = queued + __popc(pass & below);
                W.qv[at] = v;
                W.qo[at] = (uint8_t)who;
            }
            return queued + __popc(pass);
        };
        auto last_source = [&](int L, int gen) {
            return GEN && gen == GEN_LIST ? (const uint32_t*)D->cand[L] : (const uint32_t*)D->cpi_idx[L];
        };
        // Second stage: the other checks of queue entry `at` (ok lanes), finish.
        auto second_stage = [&](const LevelPlan& P, int L, const uint32_t* checks, bool ok, uint32_t at) {
            uint32_t v = 0;
            const uint32_t* c = m;
            if (ok) {
                v = W.qv[at];
                const int gen = W.qo[at] >> 5;
                c = W.m(W.qo[at] & 31);
                #pragma unroll 1
                for (int q = 0; q < L && ok; q++)  // injectivity
                    if (((P.inj >> q) & 1u) && c[q << 5] == v) ok = false;
                const int skip = gen >= 1 && gen != GEN_LIST ? P.gen[gen - 1] : -1;
                if (ok && skip >= 0) ok = tree_edge_agrees<COUNT>(g, P, c[P.par << 5], v, probes, cn);
                ok = ok && pairs_agree<COUNT>(g, c, checks, P.nchk, P.nreq, skip, v, probes, cn);
            }
            finish(ok, L, v, c);
        };
        auto count_partial = [&](const LevelPlan& P, const uint32_t* c) {
            // counting pass: the partial match is expanded once; a merge-based
            // intersection would scan the adjacency of each backward non-tree
            // neighbour's image
            cn.add(CNT_PARTIALS, 1);
            uint64_t bd = 0;
            #pragma unroll 1
            for (int q = 0; q < P.nreq; q++) {
                const uint32_t x = c[P.chk_q[q] << 5];
                bd += P.chk_dir[q] ? g.in_off[x + 1] - g.in_off[x] : g.out_off[x + 1] - g.out_off[x];
            }
            cn.add(CNT_BACK_DEG, bd);
        };
        // The last level of stored partial matches (more than FUSE_FANOUT
        // candidates each), one row after the other: its vertices in column 0, so
        // that every lane reads the same ones.
        auto run_last_rows = [&] {
            cn.cycles(CNT_CYC_TILE);
            uint64_t w = wb;
            #pragma unroll 1
            for (uint32_t r = rlo; w < we; r++) {
                const uint64_t start = ld_front(Sl + r);
                const uint64_t end = r + 1 < rhi1 ? min(we, ld_front(Sl + r + 1)) : we;
                const int32_t* const rowp = rows_l + (uint64_t)r * rw;
                __syncwarp();  // the previous row is no longer read
                if (lane <= l) *W.m(lane << 5) = (uint32_t)rowp[lane];
                __syncwarp();
                const int gen = rowp[2 * (l + 1)];
                uint32_t base = (uint32_t)rowp[2 * (l + 1) + 1];
                const uint32_t* const c0 = W.m(0);
                if (gen >= 1 && !(GEN && gen == GEN_LIST)) {
                    const int cg = LP.gen[gen - 1];
                    const uint32_t x = c0[LP.chk_q[cg] << 5];
                    base = LP.chk_dir[cg] ? __ldg(g.in_off + x) : __ldg(g.out_off + x);
                }
                if (COUNT && lane == 0 && w == start) count_partial(LP, c0);
                const FilterRow f = first_row(g, LP, c0, cw, gen);
                const uint32_t* const ids = last_source(i, gen);
                uint32_t queued = 0;
                #pragma unroll 1
                while (w < end || queued) {
                    if (w < end) {
                        uint32_t raw[LAST_WINDOWS];
#pragma unroll
                        for (int u = 0; u < LAST_WINDOWS; u++) {
                            raw[u] = 0;
                            if (w + 32 * u + lane < end) raw[u] = last_raw(LP, ids, base + (uint32_t)(w - start) + 32 * u + lane, gen);
                        }
#pragma unroll
                        for (int u = 0; u < LAST_WINDOWS; u++)
                            queued = first_stage(LP, i, queued, w + 32 * u + lane < end, raw[u], gen << 5, f);
                        __syncwarp();
                        w += 32 * LAST_WINDOWS;
                    }
                    #pragma unroll 1
                    while (queued >= 32 || (w >= end && queued)) {
                        const uint32_t take = min(queued, 32u);
                        second_stage(LP, i, cw, lane < (int)take, queued - take + lane);
                        queued -= take;
                        __syncwarp();
                        cn.iteration(true);
                    }
                }
                w = end;
            }
        };
        // The tile's items at an intermediate level (or, with LAST, of the roots
        // of a pattern of one or two nodes), compiled for the roots (level 0:
        // candidate list, 32-bit index offsets) and for stored partial matches
        // (rows, 64-bit prefixes), so that no path carries another's registers.
        auto run_tile = [&](auto last_tag, auto root_tag) {
            constexpr bool LAST = decltype(last_tag)::value;
            constexpr bool ROOT = decltype(root_tag)::value;  // expanding the roots (ROOT)
            uint32_t cur = rlo;  // row of the first work item of the iteration
            // a tile that makes partial matches of the second-to-last level
            // expands the last level of those with small fan-outs at once
            // (fused); the last level's pair checks are staged too
            const bool fuse = !LAST && k >= 3 && i == k - 2;
            if (fuse) {
                __syncwarp();
                if (lane < D->lv[k - 1].nchk) cw2[lane] = D->lv[k - 1].chk_w[lane];
                __syncwarp();
            }
            cn.cycles(CNT_CYC_TILE);
            #pragma unroll 1
            for (uint64_t w0 = wb; w0 < we; w0 += 32) {
                const uint64_t w = w0 + lane;
                bool ok = w < we;
                uint32_t v = 0;
                int32_t j = 0;
                const int32_t* rowp = nullptr;
                uint32_t r = 0;
                // Rows of this iteration's 32 work items: stored rows have fan-out
                // >= 1, so they lie in the window [cur, cur + 32); one coalesced load
                // of the window's prefixes and a 5-step shuffle search per lane. A
                // lane left at the window's end checks the next prefix and falls
                // back to a binary search (root candidates may have no fan-out).
                uint64_t sr = 0;
                if (list1) {
                    r = GEN && ok ? (uint32_t)(w / max(c1, (uint64_t)1)) : 0u;
                    sr = (uint64_t)r * c1;
                } else if (k > 1) {
                    const uint64_t widx = (uint64_t)cur + lane;
                    const uint64_t sv = widx < rhi1 ? (ROOT ? (uint64_t)__ldg(S0 + widx) : ld_front(Sl + widx))
                                                    : ~0ull;
                    int pos = 0;
                    #pragma unroll 1
                    for (int step = 16; step >= 1; step >>= 1) {
                        const uint64_t x = __shfl_sync(0xffffffffu, sv, pos + step);
                        if (x <= w) pos += step;
                    }
                    sr = __shfl_sync(0xffffffffu, sv, pos);
                    r = cur + pos;
                    if (ok && pos == 31 && r + 1 < rhi1) {
                        const uint64_t nxt = ROOT ? (uint64_t)__ldg(S0 + r + 1) : ld_front(Sl + r + 1);
                        if (nxt <= w) {
                            r = ROOT ? find_row_in(S0, r, rhi1, w) : find_row_in(Sl, r, rhi1, w);
                            sr = ROOT ? (uint64_t)__ldg(S0 + r) : ld_front(Sl + r);
                        }
                    }
                    cur = __shfl_sync(0xffffffffu, r, 31);
                }
                if (ok) {
                    cn.add(CNT_ITEMS, 1);
                    if (LAST) cn.add(CNT_ITEMS_LAST, 1);
                    if (k == 1) {
                        j = (int32_t)w;
                        v = (uint32_t)D->cand[0][j];
                    } else {
                        // the item's offset within its row's candidates, and the
                        // position of its index edge (both below 2^32: fan-outs and
                        // index lists are 32-bit)
                        const uint32_t o = (uint32_t)(w - sr);
                        uint32_t ent;
                        int choice = 0;
                        if (ROOT) {
                            // the roots' index edges are level 1's, in work-item order
                            // (or level 1's candidate list when it starts a component)
                            ent = list1 ? o : (uint32_t)w;
                            choice = list1 ? GEN_LIST : 0;
                            m[0] = (uint32_t)D->cand[0][r];
                        } else {
                            // the row's ids in 16-byte loads (rows are padded to 16 B;
                            // the columns have room for the last group), generator and
                            // index base in one 8-byte load
                            rowp = rows_l + (uint64_t)r * rw;
                            const int4* r4 = reinterpret_cast<const int4*>(rowp);
                            #pragma unroll 1
                            for (int q = 0; q <= l; q += 4) {
                                const int4 t4 = r4[q >> 2];
                                m[q << 5] = (uint32_t)t4.x;
                                m[(q + 1) << 5] = (uint32_t)t4.y;
                                m[(q + 2) << 5] = (uint32_t)t4.z;
                                m[(q + 3) << 5] = (uint32_t)t4.w;
                            }
                            const int2 gb = *reinterpret_cast<const int2*>(rowp + 2 * (l + 1));
                            choice = gb.x;
                            ent = (uint32_t)gb.y + o;
                        }
                        int skip = -1;
                        if (COUNT && o == 0) count_partial(LP, m);
                        if (choice == 0) {
                            // candidates from the index edges of the spanning-tree parent
                            if (LAST) {
                                v = __ldg(reinterpret_cast<const uint32_t*>(D->cpi_idx[i]) + ent);
                            } else {
                                const int2 e = __ldg(D->cpi_idx[i] + ent);
                                j = e.x;
                                v = (uint32_t)e.y;
                            }
                        } else if (GEN && choice == GEN_LIST) {
                            // the level starts a component: its candidate list
                            j = (int32_t)ent;
                            v = (uint32_t)__ldg(D->cand[i] + ent);
                        } else {
                            // candidates from the adjacency of the other end of a
                            // required back edge (the shorter list): keep those in
                            // C(u) and probe the spanning-tree edge instead
                            const int cg = LP.gen[choice - 1];
                            skip = cg;
                            const uint32_t x = m[LP.chk_q[cg] << 5];
                            const uint32_t p = LP.chk_dir[cg] ? __ldg(g.in_adj + __ldg(g.in_off + x) + o)
                                                              : __ldg(g.out_adj + __ldg(g.out_off + x) + o);
                            v = p >> g.lbits;
                            ok = exp_ok(LP.chk_exp[cg], (int32_t)(p & g.lmask)) &&
                                 ((__ldg(D->bm[i] + (v >> 5)) >> (v & 31)) & 1u);
                            if (ok) {
                                j = cand_rank(D->bm[i], D->rank[i], v);
                                ok = tree_edge_agrees<COUNT>(g, LP, m[LP.par << 5], v, probes, cn);
                            }
                        }
                        // injectivity, then every other pattern pair, both directions
                        #pragma unroll 1
                        for (int q = 0; q <= l && ok; q++)
                            if (((LP.inj >> q) & 1u) && m[q << 5] == v) ok = false;
                        ok = ok && pairs_agree<COUNT>(g, m, cw, nchk, LP.nreq, skip, v, probes, cn);
                    }
                    m[i << 5] = v;
                    // X pushed down: the X literals whose ends are matched at this
                    // level (before the last one; the last level checks its own)
                    if (GEN && ok && D->push_x && !LAST)
                        #pragma unroll 1
                        for (int q = 0; q < D->nx && ok; q++)
                            if (D->lit[q].lvl == i) ok = lit_holds_at(g, D->lit[q], m, i, v, COUNT ? &attr_reads : nullptr);
                }
                if (LAST) {
                    finish(ok, i, v, m);
                } else {
                    // partial match of level i: append it with its fan-out for level
                    // i+1, taken from the shortest candidate generator (dead ends,
                    // with no fan-out, are dropped)
                    uint64_t fo = 0;
                    uint32_t nbase = 0;  // where its candidates start in the generator's source
                    int gen = 0;
                    const LevelPlan& L2 = D->lv[i + 1];
                    if (ok) {
                        const int pn = L2.par;
                        if (GEN && pn < 0) {
                            // level i+1 starts a component: its whole candidate list
                            gen = GEN_LIST;
                            fo = S->ncand[i + 1];
                        } else {
                            const uint32_t ppn = pn == i ? (uint32_t)j : (ROOT ? r : (uint32_t)rowp[l + 1 + pn]);
                            const uint32_t* co = D->cpi_off[i + 1];
                            nbase = __ldg(co + ppn);
                            fo = __ldg(co + ppn + 1) - nbase;
                        }
                        #pragma unroll 1
                        for (int q = 0; q < L2.ngen; q++) {
                            const int cg = L2.gen[q];
                            const uint32_t x = m[L2.chk_q[cg] << 5];
                            const uint32_t* const off = L2.chk_dir[cg] ? g.in_off : g.out_off;
                            const uint32_t e0 = __ldg(off + x), d = __ldg(off + x + 1) - e0;
                            if (d < fo) {
                                fo = d;
                                gen = q + 1;
                                if (fuse) nbase = e0;
                            }
                        }
                    }
                    ok = ok && fo > 0;
                    bool fuse_me = fuse && ok && fo <= FUSE_FANOUT;  // expanded below, not stored
                    bool row_me = ok && !fuse_me;
                    const uint64_t packed = row_me ? ((1ull << ROW_SHIFT) | fo) : 0ull;
                    uint64_t total = 0, excl = 0;
                    if (__any_sync(0xffffffffu, row_me)) excl = warp_excl_scan(packed, lane, &total);
                    if (total) {
                        unsigned long long old = 0;
                        int full = ROWS_FIT;
                        if (lane == 0) {
                            // a full level is not counted up any further (the few warps
                            // that still do stay below the counter's 2^24 rows)
                            if (fuse) full = counter_add(__ldcg((const unsigned long long*)&S->ctr[i]), total, W.cap);
                            if (full == ROWS_FIT) {
                                old = atomicAdd((unsigned long long*)&S->ctr[i], (unsigned long long)total);
                                full = counter_add(old, total, W.cap);
                                if (full == ROWS_OUT && fuse) atomicMin((unsigned long long*)&S->row_limit, old);
                            }
                            if (full == WORK_OUT || (full && !fuse)) {
                                const uint64_t items = __ldcg((const unsigned long long*)&S->ce) - __ldcg((const unsigned long long*)&S->cb);
                                atomicExch(&S->err, __ldcg(&S->big) || items > W.cap ? DERR_WIDE : DERR_COUNTER_OVERFLOW);
                            }
                        }
                        old = __shfl_sync(0xffffffffu, old, 0);
                        // a step that fuses takes more items than the level has rows
                        // for: partial matches without a row are expanded here too
                        // (not those of a slot that has ended)
                        full = fuse ? __shfl_sync(0xffffffffu, full, 0) : ROWS_FIT;
                        if (full == ROWS_OUT) {
                            // within bounds: the step's size is a guess from the one before
                            const uint64_t work = total & WORK_MASK;
                            bool stop = __reduce_max_sync(0xffffffffu, row_me ? (uint32_t)fo : 0u) > SPILL_FANOUT;
                            if (lane == 0) {
                                stop = stop || atomicAdd((unsigned long long*)&A.sched->spilled, (unsigned long long)work) + work > FUSED_STEP_WORK;
                                if (stop) atomicExch(&S->err, DERR_WIDE);
                            }
                            if (__shfl_sync(0xffffffffu, (int)stop, 0)) full = WORK_OUT;
                            else cn.add(CNT_NO_ROW, row_me);
                        }
                        if (full) {
                            row_me = false;
                            fuse_me = ok && full == ROWS_OUT;
                        }
                        // the warp's new partial matches take rows [row0, row0 + its
                        // count) of the level's buffer, in lane order
                        if (row_me) {
                            const uint64_t row = (old >> ROW_SHIFT) + (excl >> ROW_SHIFT);
                            if (row < W.cap) {
                                cn.add(CNT_ROWS, 1);
                                // the row (ids, positions, generator, index base,
                                // padding) in 16-byte stores, four ints at a time
                                const int nw = row_width(i);
                                int32_t* dst = W.rows + row * nw;
                                #pragma unroll 1
                                for (int t = 0; t < nw; t += 4) {
                                    int32_t e4[4];
    #pragma unroll
                                    for (int c = 0; c < 4; c++) {
                                        const int idx = t + c;
                                        int32_t val = 0;
                                        if (idx <= i) {
                                            val = (int32_t)m[idx << 5];
                                        } else if (idx <= 2 * i + 1) {
                                            const int q = idx - i - 1;
                                            val = q == i ? j : (ROOT ? (int32_t)r : rowp[l + 1 + q]);
                                        } else if (idx == 2 * i + 2) {
                                            val = gen;
                                        } else if (idx == 2 * i + 3) {
                                            val = (int32_t)nbase;
                                        }
                                        e4[c] = val;
                                    }
                                    *reinterpret_cast<int4*>(dst + t) = make_int4(e4[0], e4[1], e4[2], e4[3]);
                                }
                                W.wpre[row] = (old & WORK_MASK) + (excl & WORK_MASK);
                            }
                        }
                    }
                    if (fuse) {
                        // The last level of the lanes' new partial matches with small
                        // fan-outs, by the whole warp, end to end: W.list holds the
                        // non-empty ones in order; which of them an item belongs to
                        // follows from the bits of the sequence's window at which lists
                        // start.
                        const int L = k - 1;
                        // (at most 32 x SPILL_FANOUT items)
                        const uint32_t ffo = fuse_me ? (uint32_t)fo : 0u;
                        FilterRow f{nullptr, 0};
                        if (ffo) {
                            f = first_row(g, L2, m, cw2, gen);
                            if (COUNT) count_partial(L2, m);
                        }
                        const uint32_t* const ids = last_source(L, GEN && L2.par < 0 ? GEN_LIST : 0);
                        uint32_t fin = ffo;
                        #pragma unroll 1
                        for (int d = 1; d < 32; d <<= 1) {
                            const uint32_t y = __shfl_up_sync(0xffffffffu, fin, d);
                            if (lane >= d) fin += y;
                        }
                        const uint32_t fex = fin - ffo;
                        const uint32_t ftot = __shfl_sync(0xffffffffu, fin, 31);
                        if (lane == 0 && ftot) atomicAdd((unsigned long long*)&S->st_work, (unsigned long long)ftot);
                        const uint32_t some = __ballot_sync(0xffffffffu, ffo != 0);
                        if (ffo) {
                            W.list[__popc(some & below)] = LastList{f.base, f.bits, nbase - fex};
                            W.who[__popc(some & below)] = (uint8_t)(lane | gen << 5);
                        }
                        __syncwarp();  // columns and lists are read by other lanes
                        uint32_t begun = 0, queued = 0;
                        #pragma unroll 1
                        for (uint32_t fb = 0; fb < ftot || queued;) {
                            if (fb < ftot) {
                                // which list an item is of: the lists that start up to it
                                // (bit j of starts: one starts at the window's entry j)
                                uint32_t raw[LAST_WINDOWS], own[LAST_WINDOWS];
#pragma unroll
                                for (int u = 0; u < LAST_WINDOWS; u++) {
                                    const uint32_t at = fb + 32 * u;
                                    const uint32_t starts =
                                        __reduce_or_sync(0xffffffffu, ffo && fex - at < 32u ? 1u << (fex - at) : 0u);
                                    own[u] = begun + __popc(starts & (below << 1 | 1u)) - 1;
                                    begun += __popc(starts);
                                    raw[u] = 0;
                                    if (at + lane < ftot) raw[u] = last_raw(L2, ids, at + lane + W.list[own[u]].src, W.who[own[u]] >> 5);
                                    else own[u] = 0;
                                }
#pragma unroll
                                for (int u = 0; u < LAST_WINDOWS; u++) {
                                    const LastList e = W.list[own[u]];
                                    queued = first_stage(L2, L, queued, fb + 32 * u + lane < ftot, raw[u], W.who[own[u]],
                                                         FilterRow{e.base, e.bits});
                                }
                                __syncwarp();
                                fb += 32 * LAST_WINDOWS;
                            }
                            #pragma unroll 1
                            while (queued >= 32 || (fb >= ftot && queued)) {
                                const uint32_t take = min(queued, 32u);
                                second_stage(L2, L, cw2, lane < (int)take, queued - take + lane);
                                queued -= take;
                                __syncwarp();  // the queue is written again
                            }
                        }
                    }
                }
                cn.iteration(LAST);
            }
        };
        if (last) {
            if (l == 0) run_tile(std::true_type{}, std::true_type{});
            else run_last_rows();
        } else {
            if (l == 0) run_tile(std::false_type{}, std::true_type{});
            else run_tile(std::false_type{}, std::false_type{});
        }
        if (last || i == k - 2) {
            const unsigned long long tm = __reduce_add_sync(0xffffffffu, tile_matches);
            if (lane == 0 && tm) atomicAdd((unsigned long long*)&S->n_matches, tm);
        }
        uint32_t nt = 0;
        if (lane == 0) nt = atomicAdd(&A.sched->tile_next, 1u);
        t = nwarps + __shfl_sync(0xffffffffu, nt, 0);
    }
    // probe statistics: one atomic per warp
    const unsigned long long p = __reduce_add_sync(0xffffffffu, probes);
    if (lane == 0 && p) atomicAdd((unsigned long long*)&A.sched->probes, p);
    if (COUNT) {
        cn.add(CNT_ATTR_READS, attr_reads);
        cn.flush(A.sched);
    }
}

// Start the enumeration of a slot whose index is built: level 0 holds the root
// candidates, whose work items are the index edges to level 1.
__device__ void slot_start(const SlotDesc* D, SlotState* S) {
    S->cur = 0;
    S->cursor[0] = 0;
    S->cb = S->ce = 0;
    for (int i = 0; i < D->k; i++) S->ncand[i] = *D->cand_n[i];
    S->st_cpi = 0;
    for (int i = 1; i < D->k; i++)
        if (D->lv[i].par >= 0) S->st_cpi += D->cpi_off[i][S->ncand[D->lv[i].par]];
    S->nrows[0] = S->ncand[0];
    S->big = 0;
    S->wide = 0;
    for (int l = 1; l <= D->k - 2; l++) {
        S->rows[l] = D->rows[l];
        S->wpre[l] = D->wpre[l];
        S->cap[l] = D->chunk;
    }
    S->total[0] = D->k == 1             ? (uint64_t)S->ncand[0]
                : D->lv[1].par < 0      ? (uint64_t)S->ncand[0] * S->ncand[1]  // level 1 starts a component
                                        : (uint64_t)D->cpi_off[1][S->ncand[0]];
}

// One block: finish the last step of every slot and plan the next one.
template <int CT>
__device__ void control_step(const EnumArgs& A, bool first) {
    using Scan = cub::BlockScan<unsigned long long, CT>;
    using Scan32 = cub::BlockScan<uint32_t, CT>;
    __shared__ typename Scan::TempStorage tmp;
    __shared__ typename Scan32::TempStorage tmp32;
    __shared__ unsigned long long carry_s;
    __shared__ uint32_t carry_last_s;
    __shared__ int32_t active_s;
    __shared__ int32_t expired_s;
    __shared__ unsigned long long work_s;
    if (threadIdx.x == 0) {
        carry_s = 0;
        carry_last_s = 0;
        active_s = 0;
        work_s = 0;
        // bound the whole enumeration in time: past the limit every slot stops
        const uint64_t now = globaltimer_ns();
        if (first || A.sched->t_start == 0) A.sched->t_start = now;
        expired_s = now - A.sched->t_start > A.sched->run_limit_ns;
        if (expired_s) A.sched->err = DERR_TIMEOUT;
        A.sched->spilled = 0;
    }
    // few slots left after the last step: each takes a large buffer
    const int32_t active = first ? 0 : A.sched->active;
    const bool few = A.big && !first && active <= N_BIG;
    const uint64_t share = FUSED_STEP_WORK / (uint64_t)max(active, 1);
    __syncthreads();
    for (int base = 0; base < A.n_slots; base += CT) {
        const int s = base + threadIdx.x;
        if (s < A.n_slots) {
            const SlotDesc* D = A.slots + s;
            SlotState* S = A.state + s;
            const int k = D->k;
            if (first) {
                slot_start(D, S);
            } else if (S->cur >= 0) {
                const int l = S->cur;
                S->cursor[l] = S->ce;
                S->st_steps++;
                if (k > 1 && l + 1 <= k - 2) {
                    // rows from row_limit on found no room (and were not written)
                    const uint64_t c = min(__ldcg((const unsigned long long*)&S->ctr[l + 1]),
                                           __ldcg((const unsigned long long*)&S->row_limit));
                    const uint64_t rows = c >> ROW_SHIFT;
                    if (l + 1 == k - 2 && S->ce > S->cb) {
                        // The next such step: as many items as would, like this step's,
                        // fill four fifths of the rows and lead to the slot's share of
                        // FUSED_STEP_WORK last-level items, and at most eight times as
                        // many. Items that find no row are expanded in place by the warp
                        // that has them, so that must stay the exception (and short).
                        const uint64_t items = S->ce - S->cb, cap = S->cap[l + 1];
                        const uint64_t work = (c & WORK_MASK) + (__ldcg((const unsigned long long*)&S->st_work) - S->work0);
                        uint64_t fit = min((uint64_t)LAST_LEVEL_CHUNK, 8 * max(items, cap));
                        if (rows) fit = min(fit, cap * 4 / 5 * items / rows);
                        if (work) fit = min(fit, share / work * items + share % work * items / work);
                        const bool long_lists = D->lv[k - 1].par < 0 && S->ncand[k - 1] > SPILL_FANOUT;
                        S->wide = A.narrow || long_lists ? 0 : fit;
                    }
                    if (rows > 0) {
                        S->nrows[l + 1] = rows;
                        S->total[l + 1] = c & WORK_MASK;
                        S->cursor[l + 1] = 0;
                        S->cur = l + 1;
                        S->st_rows += rows;
                    }
                }
            }
            while (S->cur >= 0 && S->cursor[S->cur] >= S->total[S->cur]) S->cur--;
            if (__ldcg(&S->err) || expired_s) S->cur = -1;
            if (S->cur < 0 && S->big) {
                atomicExch(&A.sched->big_owner[S->big - 1], 0u);
                S->big = 0;
            }
            if (S->cur >= 0) {
                const int l = S->cur;
                for (uint32_t b = 0; few && !S->big && b < N_BIG; b++)
                    if (atomicCAS(&A.sched->big_owner[b], 0u, (uint32_t)s + 1) == 0) S->big = b + 1;
                if (S->big && l + 1 <= k - 2) {  // the level to fill is empty: it moves there
                    uint8_t* const buf = A.big + (S->big - 1) * A.big_bytes;
                    S->rows[l + 1] = (int32_t*)(buf + D->big_rows[l + 1]);
                    S->wpre[l + 1] = (uint64_t*)(buf + D->big_wpre[l + 1]);
                    S->cap[l + 1] = D->big_chunk;
                }
                S->cb = S->cursor[l];
                // the last level writes no partial matches, and the one before (fused)
                // few, and expands those without a row at once, so their steps are not
                // bounded by the row buffers; a chunk of them per step left the last few
                // large GFDs of a batch with hundreds of steps of a few iterations per warp
                const uint64_t step = k == 1 || l + 1 == k - 1 ? max(D->chunk, (uint64_t)LAST_LEVEL_CHUNK)
                                      : l + 1 == k - 2         ? max(S->cap[l + 1], S->wide)
                                                               : S->cap[l + 1];
                S->ce = min(S->cb + step, S->total[l]);
                if (k > 1 && l + 1 <= k - 2) S->ctr[l + 1] = 0;
                S->row_limit = ~0ull;
                S->st_work += S->ce - S->cb;
                S->work0 = S->st_work;
                atomicAdd(&active_s, 1);
                atomicAdd(&work_s, (unsigned long long)(S->ce - S->cb));
            }
        }
    }
    __syncthreads();
    // Tile size of this step: the largest (up to A.tile) that still gives every
    // warp about four tiles, so that a step with little work (one slot at an
    // intermediate level) is spread over all warps.
    uint64_t tile = (uint64_t)A.tile;
    if (A.n_warps > 0) {
        const uint64_t per = work_s / (4ull * (uint64_t)A.n_warps);
        tile = min(tile, max((uint64_t)32, (uint64_t)((per + 31) & ~(uint64_t)31)));
    }
    // A slot whose step makes the second-to-last level's partial matches also
    // expands most of their last level inside the same tiles (fused, up to
    // FUSE_FANOUT items per partial match): its tiles are cut smaller, so that
    // no single tile holds the step's end. The step's tiles are numbered
    // heaviest first: the fusing slots', those of the other intermediate
    // levels (which store partial matches), the last level's. tile_base holds
    // three prefixes over the slots, each class from the end of the one before:
    // [0, n] fusing (F tiles), [n + 1, 2n + 1] intermediate (M), [2n + 2, 3n + 2]
    // last level. The first two counts are scanned packed in 64 bits (each total
    // is below 2^32).
    const uint64_t tile_fused = max((uint64_t)32, (tile / FUSED_TILE_DIV) & ~(uint64_t)31);
    const int n = A.n_slots;
    for (int base = 0; base < n; base += CT) {
        const int s = base + threadIdx.x;
        unsigned long long fm = 0;  // fusing << 32 | intermediate
        uint32_t nl = 0;             // last level
        if (s < n) {
            SlotState* S = A.state + s;
            if (S->cur >= 0) {
                const int k = A.slots[s].k;
                const bool fused = k >= 3 && S->cur + 1 == k - 2;
                const bool to_last = k == 1 || S->cur + 1 == k - 1;
                const uint64_t ts = fused ? tile_fused : tile;
                S->tile = (uint32_t)ts;
                const uint64_t nt = (S->ce - S->cb + ts - 1) / ts;
                if (fused) fm = nt << 32;
                else if (to_last && LAST_LEVEL_TILES_LAST) nl = (uint32_t)nt;
                else fm = nt;
            }
        }
        unsigned long long excl, total;
        Scan(tmp).ExclusiveSum(fm, excl, total);
        uint32_t lexcl, ltotal;
        Scan32(tmp32).ExclusiveSum(nl, lexcl, ltotal);
        if (s < n) {
            A.tile_base[s] = (uint32_t)((carry_s + excl) >> 32);
            A.tile_base[n + 1 + s] = (uint32_t)(carry_s + excl);  // F added below
            A.tile_base[2 * n + 2 + s] = carry_last_s + lexcl;   // F + M added below
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            carry_s += total;
            carry_last_s += ltotal;
        }
        __syncthreads();
    }
    const uint32_t nfused = (uint32_t)(carry_s >> 32), nmid = (uint32_t)carry_s, nlast = carry_last_s;
    for (int s = threadIdx.x; s < n; s += CT) {
        A.tile_base[n + 1 + s] += nfused;
        A.tile_base[2 * n + 2 + s] += nfused + nmid;
    }
    if (threadIdx.x == 0) {
        A.tile_base[n] = nfused;
        A.tile_base[2 * n + 1] = nfused + nmid;
        A.tile_base[3 * n + 2] = nfused + nmid + nlast;
        A.sched->total_tiles = nfused + nmid + nlast;
        A.sched->tile = (uint32_t)tile;
        A.sched->tile_next = 0;
        A.sched->active = active_s;
        A.sched->steps++;
        __threadfence();
    }
    __syncthreads();
}

__global__ void __launch_bounds__(CTRL_THREADS) k_control(EnumArgs A, int first) {
    control_step<CTRL_THREADS>(A, first != 0);
}

template <int NT, int MINB, bool GEN>
__global__ void __launch_bounds__(NT, MINB) k_expand(EnumArgs A) {
    expand_warps<NT, GEN, false>(A);
}

// Bounded grid barrier (cooperative launch guarantees co-residency): the last
// arriving block bumps the generation; the others wait for it, up to
// sched->timeout_ns, after which they record DERR_TIMEOUT and give up.
__device__ bool grid_barrier(Sched* s) {
    __syncthreads();
    __shared__ int ok_s;
    if (threadIdx.x == 0) {
        volatile uint32_t* genp = &s->bar_gen;
        const uint32_t gen = *genp;
        __threadfence();
        const uint32_t arrived = atomicAdd(&s->bar_count, 1u);
        int ok = 1;
        if (arrived == gridDim.x - 1) {
            atomicExch(&s->bar_count, 0u);
            __threadfence();
            atomicAdd(&s->bar_gen, 1u);
        } else {
            const uint64_t t0 = globaltimer_ns();
            while (*genp == gen) {
                if (*(volatile int32_t*)&s->err) {
                    ok = 0;
                    break;
                }
                if (globaltimer_ns() - t0 > s->timeout_ns) {
                    atomicExch(&s->err, DERR_TIMEOUT);
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

template <int NT, int MINB, bool GEN, bool COUNT = false>
__global__ void __launch_bounds__(NT, MINB) k_persistent(EnumArgs A) {
    for (;;) {
        expand_warps<NT, GEN, COUNT>(A);
        if (!grid_barrier(A.sched)) return;
        if (blockIdx.x == 0) control_step<NT>(A, false);
        if (!grid_barrier(A.sched)) return;
        if (*(volatile int32_t*)&A.sched->active == 0) return;
    }
}

template <int NT, int MINB, bool GEN, bool COUNT = false>
int launch_persistent(const EnumArgs& a, cudaStream_t st, int64_t* launches) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = warp_shared_bytes(a.kmax) * (NT / 32);
    cudaError_t e = cudaFuncSetAttribute(k_persistent<NT, MINB, GEN, COUNT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(warp_shared_bytes(MAXK) * (NT / 32)));
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_persistent<NT, MINB, GEN, COUNT>, NT, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    if (per_sm < 1) {
        set_error(GFD_ERR_CUDA, "persistent enumeration kernel cannot be resident");
        return GFD_ERR_CUDA;
    }
    const int grid = sms * per_sm;
    EnumArgs args = a;
    args.n_warps = grid * (NT / 32);
    args.columns = (uint32_t)column_words(a.kmax);
    void* params[] = {&args};
    e = cudaLaunchCooperativeKernel((const void*)k_persistent<NT, MINB, GEN, COUNT>, dim3(grid), dim3(NT), params, smem,
                                    st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaLaunchCooperativeKernel");
    if (launches) *launches += 1;
    return GFD_OK;
}

template <int NT, int MINB, bool GEN>
int expand_grid(size_t smem) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(k_expand<NT, MINB, GEN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(warp_shared_bytes(MAXK) * (NT / 32)));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_expand<NT, MINB, GEN>, NT, smem);
    return sms * std::max(per_sm, 1);
}

template <int NT, int MINB, bool GEN>
int host_loop(const EnumArgs& a0, bool use_graph, cudaStream_t st, int64_t* launches) {
    const size_t smem = warp_shared_bytes(a0.kmax) * (NT / 32);
    const int grid = expand_grid<NT, MINB, GEN>(smem);
    EnumArgs a = a0;
    a.n_warps = grid * (NT / 32);
    a.columns = (uint32_t)column_words(a0.kmax);
    int32_t* h_active = nullptr;
    cudaError_t e = cudaMallocHost(&h_active, sizeof(int32_t));
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocHost");
    const int per_check = 8;
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t graph = nullptr;
    int rc = GFD_OK;
    if (use_graph) {
        e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            for (int it = 0; it < per_check; it++) {
                k_expand<NT, MINB, GEN><<<grid, NT, smem, st>>>(a);
                k_control<<<1, CTRL_THREADS, 0, st>>>(a, 0);
            }
            e = cudaStreamEndCapture(st, &graph);
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
        if (e != cudaSuccess) {
            cudaFreeHost(h_active);
            if (graph) cudaGraphDestroy(graph);
            return cuda_fail(e, "CUDA graph capture of the enumeration steps");
        }
    }
    for (int64_t round = 0;; round++) {
        if (use_graph) {
            e = cudaGraphLaunch(exec, st);
            if (launches) *launches += 2 * per_check;
        } else {
            for (int it = 0; it < per_check; it++) {
                k_expand<NT, MINB, GEN><<<grid, NT, smem, st>>>(a);
                k_control<<<1, CTRL_THREADS, 0, st>>>(a, 0);
            }
            e = cudaGetLastError();
            if (launches) *launches += 2 * per_check;
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(h_active, &a.sched->active, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "enumeration step");
            break;
        }
        if (*h_active == 0) break;
    }
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    cudaFreeHost(h_active);
    return rc;
}

// one thread per violation record: append it to its GFD's list
__global__ void k_split(const SlotDesc* slots, const int32_t* arena, uint64_t n, int32_t stride,
                        int32_t* const* lists, unsigned long long* cursor) {
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < n; r += (uint64_t)gridDim.x * blockDim.x) {
        const int32_t* rec = arena + r * stride;
        const int s = rec[0];
        const int k = slots[s].k;
        // one atomic per group of lanes with the same slot (records of one
        // slot arrive in runs, so a warp usually needs one or two)
        const int lane = threadIdx.x & 31;
        const uint32_t peers = __match_any_sync(__activemask(), s);
        const int leader = __ffs(peers) - 1;
        unsigned long long base = 0;
        if (lane == leader) base = atomicAdd(&cursor[s], (unsigned long long)__popc(peers));
        base = __shfl_sync(peers, base, leader);
        const uint64_t pos = base + __popc(peers & ((1u << lane) - 1u));
        int32_t* dst = lists[s] + pos * k;
        for (int q = 0; q < k; q++) dst[q] = rec[1 + q];
    }
}

__global__ void k_mark_idle(SlotState* state, int n) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) state[s].cur = -1;
}

// Slots admitted between steps: start them (the next control step plans their
// first chunk), finishing at once when level 0 has no work. The slot ids
// travel in the kernel parameters.
struct SlotIds {
    int n;
    int v[64];
};

__global__ void k_init_slots(EnumArgs A, SlotIds ids) {
    const int i = threadIdx.x;
    if (i >= ids.n) return;
    const int s = ids.v[i];
    SlotState* S = A.state + s;
    slot_start(A.slots + s, S);
    if (S->total[0] == 0) S->cur = -1;
}

}  // namespace

int mark_idle(SlotState* state, int n, cudaStream_t st) {
    k_mark_idle<<<std::max(1, (n + 255) / 256), 256, 0, st>>>(state, n);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GFD_OK : cuda_fail(e, "k_mark_idle");
}

int init_slots(const EnumArgs& a, const int* host_ids, int n, cudaStream_t st) {
    for (int b = 0; b < n; b += 64) {
        SlotIds ids{};
        ids.n = std::min(64, n - b);
        for (int i = 0; i < ids.n; i++) ids.v[i] = host_ids[b + i];
        k_init_slots<<<1, 64, 0, st>>>(a, ids);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GFD_OK : cuda_fail(e, "k_init_slots");
}

int launch_split(const SlotDesc* slots, const int32_t* arena, uint64_t n, int32_t stride, int32_t* const* lists,
                 unsigned long long* cursor, cudaStream_t st) {
    const int grid = (int)std::min<uint64_t>((n + 255) / 256, (uint64_t)device_sms() * 16);
    k_split<<<std::max(grid, 1), 256, 0, st>>>(slots, arena, n, stride, lists, cursor);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GFD_OK : cuda_fail(e, "k_split");
}

namespace {

template <int NT, int MINB, bool GEN>
int capture_steps_t(const EnumArgs& a0, int steps, cudaStream_t st, cudaGraph_t* graph, cudaGraphExec_t* exec) {
    const size_t smem = warp_shared_bytes(a0.kmax) * (NT / 32);
    const int grid = expand_grid<NT, MINB, GEN>(smem);
    EnumArgs a = a0;
    a.n_warps = grid * (NT / 32);
    a.columns = (uint32_t)column_words(a0.kmax);
    cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        for (int it = 0; it < steps; it++) {
            k_expand<NT, MINB, GEN><<<grid, NT, smem, st>>>(a);
            k_control<<<1, CTRL_THREADS, 0, st>>>(a, 0);
        }
        e = cudaStreamEndCapture(st, graph);
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(exec, *graph, 0);
    if (e != cudaSuccess) return cuda_fail(e, "CUDA graph capture of the enumeration steps");
    return GFD_OK;
}

template <int NT, int MINB, bool GEN>
int run_variant(const EnumArgs& a, bool persistent, bool use_graph, cudaStream_t st, int64_t* launches) {
    return persistent ? launch_persistent<NT, MINB, GEN>(a, st, launches) : host_loop<NT, MINB, GEN>(a, use_graph, st, launches);
}

}  // namespace

// Kernel variants: threads per block and the minimum resident blocks per SM the
// compiler must allow (which caps registers per thread).
int variant_threads(int v) {
    switch (v) {
        case 3: return 128;
        case 5: return 512;
        default: return 256;
    }
}

int capture_steps(const EnumArgs& a, int variant, int steps, cudaStream_t st, cudaGraph_t* graph,
                  cudaGraphExec_t* exec) {
    // a session admits any request later: the general expansion
    constexpr bool GEN = true;
    switch (variant) {
        case 1: return capture_steps_t<256, 6, GEN>(a, steps, st, graph, exec);
        case 2: return capture_steps_t<256, 8, GEN>(a, steps, st, graph, exec);
        case 3: return capture_steps_t<128, 12, GEN>(a, steps, st, graph, exec);
        case 4: return capture_steps_t<256, 5, GEN>(a, steps, st, graph, exec);
        case 5: return capture_steps_t<512, 3, GEN>(a, steps, st, graph, exec);
        default: return capture_steps_t<256, 4, GEN>(a, steps, st, graph, exec);
    }
}

namespace {

template <bool GEN>
int run_any_variant(const EnumArgs& a, bool persistent, bool use_graph, int variant, cudaStream_t st,
                    int64_t* launches) {
    switch (variant) {
        case 1: return run_variant<256, 6, GEN>(a, persistent, use_graph, st, launches);
        case 2: return run_variant<256, 8, GEN>(a, persistent, use_graph, st, launches);
        case 3: return run_variant<128, 12, GEN>(a, persistent, use_graph, st, launches);
        case 4: return run_variant<256, 5, GEN>(a, persistent, use_graph, st, launches);
        case 5: return run_variant<512, 3, GEN>(a, persistent, use_graph, st, launches);
        default: return run_variant<256, 4, GEN>(a, persistent, use_graph, st, launches);
    }
}

}  // namespace

int enum_init(const EnumArgs& a, cudaStream_t st) {
    k_control<<<1, CTRL_THREADS, 0, st>>>(a, 1);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GFD_OK : cuda_fail(e, "k_control");
}

int enum_run(const EnumArgs& a, bool persistent, bool use_graph, int variant, bool general, cudaStream_t st,
             cudaEvent_t ev0, cudaEvent_t ev1, int64_t* launches, bool count) {
    if (ev0) cudaEventRecord(ev0, st);
    const int rc = count     ? launch_persistent<256, 4, true, true>(a, st, launches)
                 : general ? run_any_variant<true>(a, persistent, use_graph, variant, st, launches)
                           : run_any_variant<false>(a, persistent, use_graph, variant, st, launches);
    if (ev1) cudaEventRecord(ev1, st);
    return rc;
}

}  // namespace gfd
