// Compact path index construction (Section III.B, step 1).
//
//   k_filter   step 1a-1b: candidates by label and degree (and self-loop, and
//              pushed-down constant X literals), one coalesced pass over vertex
//              data for all filter keys;
//   k_scatter  step 1c: mark vertices adjacent (in the direction and with the
//              label of a pattern edge) to the candidates of another level;
//   k_refine   step 1c: keep the candidates that are marked, and those with such
//              a neighbour among the candidates of another level (early exit at
//              the first one); top-down and bottom-up use whichever of marking
//              and looking is cheaper;
//   k_compact  bitmap -> exclusive popcount prefix (O(1) rank) + sorted list;
//   k_cpi_*    step 1d: for each spanning-tree edge, the index edges from
//              every parent candidate to the positions of its child candidates.
//
// Every launch processes a table of jobs. Candidates are read from bitmaps, so
// refinement needs no lists: a launch per level and direction (two with marks).
// Which vertices can be in a bitmap is known on the host (a label's range in each
// degree class), so the jobs' shares of a launch are laid out there (ScanRange)
// and no kernel counts or scans between two steps of the refinement. Before, with
// a list per level and step and its compaction in between (up to seven launches
// per level and direction), a triangle with a chain on 1M vertices took 0.50 ms
// of refinement in 47 launches, and 16 requests on 1M vertices 7.3 ms in 690; now
// 0.21 ms in 10 and 3.5 ms in 194.
#include <cub/cub.cuh>

#include <algorithm>
#include <map>
#include <mutex>

#include "engine.h"

namespace gfd {

namespace {

constexpr int FILTER_THREADS = 256;
constexpr int COMPACT_THREADS = 256;
constexpr uint32_t COMPACT_WORDS = 256;   // bitmap words per chunk of the compaction
constexpr uint32_t CPI_CHUNK = 1024;      // counts per chunk of the index offsets
constexpr int WARP_KERNEL_THREADS = 256;

__device__ __forceinline__ uint64_t gwarp_id() {
    return (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
}
__device__ __forceinline__ uint64_t nwarps_total() { return ((uint64_t)gridDim.x * blockDim.x) >> 5; }

__global__ void k_filter(DevGraph g, const FilterKey* __restrict__ keys, int nkeys, uint32_t* __restrict__ out) {
    extern __shared__ FilterKey sk[];
    for (int i = threadIdx.x; i < nkeys; i += blockDim.x) sk[i] = keys[i];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (uint64_t w = gwarp_id(); w < g.nwords; w += nwarps_total()) {
        const uint32_t v = (uint32_t)w * 32 + lane;
        const bool valid = v < (uint32_t)g.n;
        uint32_t vi = 0, dout = 0, din = 0;
        if (valid) {
            vi = g.vinfo[v];
            dout = g.out_off[v + 1] - g.out_off[v];
            din = g.in_off[v + 1] - g.in_off[v];
        }
        const int32_t L = (int32_t)(vi & 0xffffu);
        const bool has_self = (vi >> 16) != 0;
        const int32_t self_lab = (int32_t)(vi >> 16) - 1;
        dout -= has_self;
        din -= has_self;
        for (int k = 0; k < nkeys; k++) {
            const FilterKey& key = sk[k];  // fields read from shared memory as needed
            bool self_ok = key.self_exp == EXP_SKIP ? true
                         : key.self_exp == EXP_NONE ? !has_self
                         : key.self_exp == EXP_ANY  ? has_self
                                                    : (has_self && self_lab == key.self_exp);
            bool p = valid && label_ok(key.label, L) && dout >= key.dout_min && din >= key.din_min && self_ok;
            for (int t = 0; t < key.n_attr; t++) {  // pushed-down constant X literals
                const int32_t va = p ? g.attrs[(uint64_t)key.attr_a[t] * g.n + v] : GFD_ATTR_ABSENT;
                p = p && va != GFD_ATTR_ABSENT && va == key.attr_c[t];
            }
            uint32_t b = __ballot_sync(0xffffffffu, p);
            if (lane == 0) out[(uint64_t)k * g.nwords + w] = b;
        }
    }
}

// Compaction in two passes over (job, chunk) items so that even one job uses
// the whole GPU: k_compact_sums counts set bits per chunk of COMPACT_WORDS
// words; k_compact_write adds the counts of the preceding chunks, scans its own
// chunk and writes rank[w] (set bits before word w) and the candidate list.
__global__ void __launch_bounds__(COMPACT_THREADS) k_compact_sums(DevGraph g, const CompactJob* __restrict__ jobs,
                                                                  int njobs, uint32_t nchunks) {
    using Reduce = cub::BlockReduce<uint32_t, COMPACT_THREADS>;
    __shared__ typename Reduce::TempStorage tmp;
    for (uint64_t it = blockIdx.x; it < (uint64_t)njobs * nchunks; it += gridDim.x) {
        const CompactJob& J = jobs[it / nchunks];
        const uint32_t c = (uint32_t)(it % nchunks);
        uint32_t cnt = 0;
        for (uint32_t w = c * COMPACT_WORDS + threadIdx.x; w < min(g.nwords, (c + 1) * COMPACT_WORDS);
             w += COMPACT_THREADS)
            cnt += __popc(J.bm[w]);
        cnt = Reduce(tmp).Sum(cnt);
        if (threadIdx.x == 0) J.csum[c] = cnt;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(COMPACT_THREADS) k_compact_write(DevGraph g, const CompactJob* __restrict__ jobs,
                                                                   int njobs, uint32_t nchunks) {
    using Scan = cub::BlockScan<uint32_t, COMPACT_THREADS>;
    using Reduce = cub::BlockReduce<uint32_t, COMPACT_THREADS>;
    __shared__ union {
        typename Scan::TempStorage scan;
        typename Reduce::TempStorage reduce;
    } tmp;
    __shared__ uint32_t base_s;
    constexpr int WPT = COMPACT_WORDS / COMPACT_THREADS;  // words per thread
    for (uint64_t it = blockIdx.x; it < (uint64_t)njobs * nchunks; it += gridDim.x) {
        const CompactJob& J = jobs[it / nchunks];
        const uint32_t c = (uint32_t)(it % nchunks);
        uint32_t before = 0;
        for (uint32_t q = threadIdx.x; q < c; q += COMPACT_THREADS) before += J.csum[q];
        before = Reduce(tmp.reduce).Sum(before);
        if (threadIdx.x == 0) base_s = before;
        __syncthreads();
        const uint32_t w0 = c * COMPACT_WORDS + threadIdx.x * WPT;
        uint32_t words[WPT];
        uint32_t cnt = 0;
        for (int q = 0; q < WPT; q++) {
            words[q] = w0 + q < g.nwords ? J.bm[w0 + q] : 0u;
            cnt += __popc(words[q]);
        }
        uint32_t excl, total;
        Scan(tmp.scan).ExclusiveSum(cnt, excl, total);
        uint32_t r = base_s + excl;
        uint32_t first[WPT];  // list position of each word's first vertex
#pragma unroll
        for (int q = 0; q < WPT; q++) {
            first[q] = r;
            if (w0 + q < g.nwords) J.rank[w0 + q] = r;
            r += __popc(words[q]);
        }
        // the list, by the whole warp: one word with candidates at a time, a lane
        // per bit, so that the stores of a word are next to each other
        int32_t* const cand = J.cand;
        const uint32_t lane = threadIdx.x & 31;
#pragma unroll
        for (int q = 0; q < WPT && cand; q++)
            for (uint32_t some = __ballot_sync(0xffffffffu, words[q] != 0); some; some &= some - 1) {
                const int src = __ffs(some) - 1;
                const uint32_t x = __shfl_sync(0xffffffffu, words[q], src), at = __shfl_sync(0xffffffffu, first[q], src);
                const uint32_t w = __shfl_sync(0xffffffffu, w0 + q, src);
                if ((x >> lane) & 1u) cand[at + __popc(x & ((1u << lane) - 1u))] = (int32_t)(w * 32 + lane);
            }
        if (c == nchunks - 1 && threadIdx.x == 0) *J.count = base_s + total;
        __syncthreads();
    }
}

// The adjacency kernels below give the lanes of a warp a candidate each; the warp
// then scans its lists end to end as one sequence, 32 x FLAT entries at a time
// (scan_flat). A hub's list is scanned by a block.
//
// These scans are bound by latency (a random adjacency line, then a random
// bitmap word, from L2 or HBM) and by balance. A lane that scans its own list
// leaves the warp waiting for its longest list with few loads in flight; a warp
// that happens to get 32 long lists keeps the launch waiting. End to end every
// lane has FLAT loads in flight whatever the degrees, and by degree classes a warp
// of a small launch gets no more than 2048 entries at a time (one vertex of up to
// 2048, 8 of up to 256, 32 of up to 32), one of a large launch no more than 8192 (4,
// 32 and 32 vertices; see scan_units).
constexpr int FLAT = 4;
constexpr int MAX_WORDS = 32;  // most bitmap words per warp item of the last class
// Resident blocks per SM the scanning kernels are compiled for; at 6 the
// refinement's registers spill (a triangle with a chain on 1M vertices: 0.22 ms of
// refinement at 5, 0.35 ms at 6).
constexpr int SCAN_BLOCKS = 6;
constexpr int REFINE_BLOCKS = 5;

// Entries of the aligned quad at b < e1 that lie in [e0, e1), as a mask.
__device__ __forceinline__ uint32_t quad_mask(uint32_t b, uint32_t e0, uint32_t e1) {
    uint32_t m = 15u;
    if (b < e0) m &= m << (e0 - b);
    if (e1 - b < 4u) m &= (1u << (e1 - b)) - 1u;
    return m;
}

// Of the entries m of the aligned quad at b, those with an allowed edge label
// whose neighbour is in bm; x receives the neighbours, w their bitmap words.
__device__ __forceinline__ uint32_t quad_hits(const DevGraph& g, const uint32_t* adj, uint32_t b, uint32_t m, int32_t lab,
                                              const uint32_t* bm, uint32_t (&x)[4], uint32_t (&w)[4]) {
    const uint4 p4 = __ldg(reinterpret_cast<const uint4*>(adj + b));
    const uint32_t p[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
    for (int t = 0; t < 4; t++) {
        x[t] = p[t] >> g.lbits;
        const bool ok = ((m >> t) & 1u) && label_ok(lab, (int32_t)(p[t] & g.lmask));
        w[t] = ok ? __ldg(bm + (x[t] >> 5)) : 0u;
    }
    uint32_t h = 0;
#pragma unroll
    for (int t = 0; t < 4; t++) h |= ((w[t] >> (x[t] & 31)) & 1u) << t;
    return h;
}

// The adjacency a job scans.
struct AdjRef {
    const uint32_t* off;
    const uint32_t* adj;
};
__device__ __forceinline__ AdjRef adj_ref(const DevGraph& g, bool out) {
    return out ? AdjRef{g.out_off, g.out_adj} : AdjRef{g.in_off, g.in_adj};
}

// The warp's 32 lists, lane i holding [e0, e1) (empty for e0 = e1), scanned end
// to end. f(hit, x, w, owner, window) is called by all lanes for every window of
// 32 entries, in order: whether the lane's entry has allowed labels and a
// neighbour x in bm (w: its bitmap word), and the lane whose list it is from;
// window: position of the window in the sequence. slots: the warp's 32 int2 in
// shared memory. ex: where the lane's list starts in the sequence (for f).
template <typename F>
__device__ __forceinline__ void scan_flat(const DevGraph& g, const AdjRef& A, uint32_t e0, uint32_t len, uint32_t ex,
                                          uint32_t total, int32_t lab, const uint32_t* bm, int2* slots, int lane,
                                          F&& f) {
    // the non-empty lists in order: (position in adj - position in the sequence, lane)
    const uint32_t some = __ballot_sync(0xffffffffu, len != 0);
    if (len) slots[__popc(some & ((1u << lane) - 1u))] = make_int2((int32_t)(e0 - ex), lane);
    __syncwarp();
    const uint32_t upto = 0xffffffffu >> (31 - lane);
    uint32_t begun = 0;  // lists that start before the window
    for (uint32_t base = 0; base < total; base += 32 * FLAT) {
        uint32_t p[FLAT], w[FLAT];
        int owner[FLAT];
#pragma unroll
        for (int u = 0; u < FLAT; u++) {
            const uint32_t wb = base + 32u * u;
            // bit i: a list starts at the window's i-th entry
            const uint32_t starts = __reduce_or_sync(0xffffffffu, len && ex - wb < 32u ? 1u << (ex - wb) : 0u);
            const uint32_t o = begun + __popc(starts & upto) - 1;
            begun += __popc(starts);
            owner[u] = -1;
            p[u] = 0;
            if (wb + lane < total) {
                const int2 s = slots[o];
                const uint32_t e = wb + lane + (uint32_t)s.x;
                p[u] = __ldg(A.adj + e);
                owner[u] = s.y;
            }
        }
#pragma unroll
        for (int u = 0; u < FLAT; u++)
            w[u] = owner[u] >= 0 && label_ok(lab, (int32_t)(p[u] & g.lmask)) ? __ldg(bm + ((p[u] >> g.lbits) >> 5)) : 0u;
#pragma unroll
        for (int u = 0; u < FLAT; u++) {
            const uint32_t x = p[u] >> g.lbits;
            f((bool)((w[u] >> (x & 31)) & 1u), x, w[u], owner[u], base + 32u * u);
        }
        if (total - base <= 32u * FLAT) break;  // (base + 32 FLAT could wrap)
    }
    __syncwarp();  // slots are written again by the next scan
}

// Exclusive warp scan of the lanes' list lengths (their sum is below 2^32: lists
// of different vertices).
__device__ __forceinline__ uint32_t list_starts(uint32_t len, int lane, uint32_t* total) {
    uint32_t incl = len;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    *total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - len;
}

// the job that holds item it of the launch (first: items of the earlier jobs);
// *at: its number within the job
__device__ __forceinline__ int job_of(const uint32_t* first, int njobs, uint32_t it, uint32_t* at) {
    int lo = 0, hi = njobs;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(first + mid) <= it) lo = mid;
        else hi = mid;
    }
    *at = it - __ldg(first + lo);
    return lo;
}

// The vertices [a, b) of a range's warp item `it` (a = b: none).
__device__ __forceinline__ void item_range(const ScanRange& R, uint32_t it, const ScanLaunch& l, uint32_t* a,
                                           uint32_t* b) {
    const bool flat = R.flat;
#pragma unroll
    for (int c = 0; c < N_CLASS; c++) {
        if (c == 0 && !flat) continue;
        const int unit = flat ? FLAT_UNIT : l.unit[c];
        const uint32_t lo = R.lo[c], hi = R.hi[c], items = scan_items(lo, hi, unit);
        if (it < items) {
            const uint64_t from = (uint64_t)((lo >> unit) + it) << unit;
            *a = max(lo, (uint32_t)from);
            *b = (uint32_t)min((unsigned long long)hi, (unsigned long long)from + (1ull << unit));
            return;
        }
        it -= items;
    }
    *a = *b = 0;
}

// The word at w (lane's) of an item's vertices [a, b), bits outside cleared.
__device__ __forceinline__ uint32_t item_mask(uint32_t w, uint32_t a, uint32_t b) {
    uint32_t m = 0xffffffffu;
    if (w == a >> 5) m &= m << (a & 31);
    if (w == (b - 1) >> 5) m &= 0xffffffffu >> (31 - ((b - 1) & 31));
    return m;
}

// The set bits of the warp's words x (lane j < nw holding word j) as a list of
// word << 5 | bit in shared memory; returns how many.
__device__ __forceinline__ uint32_t expand_bits(uint32_t x, uint16_t* list, int lane) {
    uint32_t n = 0;
    for (uint32_t some = __ballot_sync(0xffffffffu, x != 0); some; some &= some - 1) {
        const int j = __ffs(some) - 1;
        const uint32_t y = __shfl_sync(0xffffffffu, x, j);
        if ((y >> lane) & 1u) list[n + __popc(y & ((1u << lane) - 1u))] = (uint16_t)(j << 5 | lane);
        n += __popc(y);
    }
    __syncwarp();
    return n;
}

// Counting pass: add this thread's scanned candidates and adjacency entries to
// the run's counters (all lanes of the warp call it; one atomic per warp).
template <bool COUNT>
__device__ __forceinline__ void scan_flush(ScanCount scan, uint64_t cands, uint64_t entries) {
    if (!COUNT) return;
    for (int d = 16; d >= 1; d >>= 1) {
        cands += __shfl_xor_sync(0xffffffffu, cands, d);
        entries += __shfl_xor_sync(0xffffffffu, entries, d);
    }
    if ((threadIdx.x & 31) == 0) {
        if (cands) atomicAdd(&scan[0], (unsigned long long)cands);
        if (entries) atomicAdd(&scan[1], (unsigned long long)entries);
    }
}

// A hub's list [e0, e1) scanned by the block: f(hits, x, w) per quad, where a
// thread takes HUB_QUADS quads in a row per round; stop() is asked after every
// round by all threads.
constexpr int HUB_QUADS = 4;
template <typename F, typename Stop>
__device__ __forceinline__ void scan_block(const DevGraph& g, const uint32_t* adj, uint32_t e0, uint32_t e1, int32_t lab,
                                           const uint32_t* bm, F&& f, Stop&& stop) {
    constexpr uint32_t ROUND = 4 * HUB_QUADS * WARP_KERNEL_THREADS;
    for (uint64_t r = e0 & ~3u; r < e1; r += ROUND) {  // block-uniform bounds
#pragma unroll
        for (int q = 0; q < HUB_QUADS; q++) {
            const uint64_t b = r + 4u * (HUB_QUADS * threadIdx.x + q);
            uint32_t x[4], w[4], h = 0;
            if (b < e1) h = quad_hits(g, adj, (uint32_t)b, quad_mask((uint32_t)b, e0, e1), lab, bm, x, w);
            if (h) f(q, h, x, w);
        }
        if (stop()) return;
    }
}

// Mark vertex x. Popular vertices are reached over and over, and numbered next to
// each other, so their words would take most of the atomics: a look (possibly
// at an old copy in L1, which only costs a needless atomic) leaves those out.
__device__ __forceinline__ void mark(uint32_t* marks, uint32_t x) {
    uint32_t* const w = marks + (x >> 5);
    const uint32_t b = 1u << (x & 31);
    if (!(__ldca(w) & b)) atomicOr(w, b);
}

// Shared memory of a warp in the scanning kernels.
struct ScanShared {
    int2 slots[WARP_KERNEL_THREADS];
    uint16_t list[WARP_KERNEL_THREADS / 32][32 * MAX_WORDS];  // an item's candidates
};

template <bool COUNT>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS, SCAN_BLOCKS) k_scatter(DevGraph g, const ScatterJob* __restrict__ jobs,
                                                                 int njobs, ScanLaunch l, ScanCount scan) {
    __shared__ ScanShared sh;
    const int lane = threadIdx.x & 31;
    int2* const slots = sh.slots + (threadIdx.x & ~31);
    uint16_t* const list = sh.list[threadIdx.x >> 5];
    uint64_t sc = 0, se = 0;
    for (uint32_t it = blockIdx.x; it < l.hubs; it += gridDim.x) {
        uint32_t at;
        const ScatterJob& J = jobs[job_of(l.hub_first, njobs, it, &at)];
        const uint32_t v = J.r.lo[0] + at;
        if (!((J.r.bm[v >> 5] >> (v & 31)) & 1u)) continue;
        const AdjRef A = adj_ref(g, J.scan_out);
        const uint32_t e0 = A.off[v], e1 = A.off[v + 1];
        if (threadIdx.x == 0) sc += e1 > e0, se += e1 - e0;
        uint32_t* const marks = J.marks;
        scan_block(g, A.adj, e0, e1, J.lab, J.filter,
                   [&](int, uint32_t h, const uint32_t (&x)[4], const uint32_t (&)[4]) {
#pragma unroll
                       for (int c = 0; c < 4; c++)
                           if ((h >> c) & 1u) mark(marks, x[c]);
                   },
                   [] { return false; });
    }
    for (uint64_t it = gwarp_id(); it < l.items; it += nwarps_total()) {
        uint32_t item, va, vb;
        const ScatterJob& J = jobs[job_of(l.first, njobs, (uint32_t)it, &item)];
        item_range(J.r, item, l, &va, &vb);
        const uint32_t w0 = va >> 5, nw = (vb + 31) / 32 - w0;
        const uint32_t x = lane < (int)nw ? J.r.bm[w0 + lane] & item_mask(w0 + lane, va, vb) : 0u;
        if (!__any_sync(0xffffffffu, x != 0)) continue;
        const uint32_t n = expand_bits(x, list, lane);
        const AdjRef A = adj_ref(g, J.scan_out);
        uint32_t* const marks = J.marks;
        for (uint32_t i = 0; i < n; i += 32) {
            uint32_t e0 = 0, e1 = 0;
            if (i + lane < n) {
                const uint32_t v = w0 * 32 + list[i + lane];
                e0 = A.off[v];
                e1 = A.off[v + 1];
            }
            sc += e1 > e0;
            se += e1 - e0;
            uint32_t total;
            const uint32_t ex = list_starts(e1 - e0, lane, &total);
            scan_flat(g, A, e0, e1 - e0, ex, total, J.lab, J.filter, slots, lane,
                      [&](bool hit, uint32_t y, uint32_t, int, uint32_t) {
                          if (hit) mark(marks, y);
                      });
        }
        __syncwarp();  // list is written again
    }
    scan_flush<COUNT>(scan, sc, se);
}

// A constraint on neighbours of any vertex label hits often: each lane first
// tries its own list's first quad, and only lists without a hit there are
// scanned end to end.
template <bool COUNT>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS, REFINE_BLOCKS) k_refine(DevGraph g, const RefineJob* __restrict__ jobs, int njobs,
                                                                ScanLaunch l, ScanCount scan) {
    __shared__ ScanShared sh;
    __shared__ uint8_t s_hit[WARP_KERNEL_THREADS];
    __shared__ uint32_t s_keep[WARP_KERNEL_THREADS / 32][MAX_WORDS];
    const int lane = threadIdx.x & 31;
    int2* const slots = sh.slots + (threadIdx.x & ~31);
    uint16_t* const list = sh.list[threadIdx.x >> 5];
    uint8_t* const found = s_hit + (threadIdx.x & ~31);
    uint32_t* const kept = s_keep[threadIdx.x >> 5];
    uint64_t sc = 0, se = 0;
    for (uint32_t it = blockIdx.x; it < l.hubs; it += gridDim.x) {
        uint32_t at;
        const RefineJob& J = jobs[job_of(l.hub_first, njobs, it, &at)];
        const uint32_t v = J.r.lo[0] + at;
        uint32_t x = J.r.bm[v >> 5];
        for (int m = 0; m < J.nmarks; m++) x &= J.marks[m][v >> 5];
        bool keep = (x >> (v & 31)) & 1u;
        for (int c = 0; c < J.ncon && keep; c++) {  // block-uniform
            const AdjRef A = adj_ref(g, J.con_dir[c]);
            const uint32_t e0 = A.off[v], e1 = A.off[v + 1];
            if (threadIdx.x == 0) sc++, se += e1 - e0;
            bool hit = false;
            keep = false;
            scan_block(g, A.adj, e0, e1, J.con_lab[c], J.con_bm[c],
                       [&](int, uint32_t, const uint32_t (&)[4], const uint32_t (&)[4]) { hit = true; },
                       [&] { return keep = __syncthreads_or(hit); });
        }
        if (keep && threadIdx.x == 0) atomicOr(&J.out[v >> 5], 1u << (v & 31));
    }
    for (uint64_t it = gwarp_id(); it < l.items; it += nwarps_total()) {
        uint32_t item, va, vb;
        const RefineJob& J = jobs[job_of(l.first, njobs, (uint32_t)it, &item)];
        item_range(J.r, item, l, &va, &vb);
        const uint32_t w0 = va >> 5, nw = (vb + 31) / 32 - w0;
        uint32_t x = 0;
        if (lane < (int)nw) {
            x = J.r.bm[w0 + lane] & item_mask(w0 + lane, va, vb);
            for (int m = 0; m < J.nmarks; m++) x &= J.marks[m][w0 + lane];
        }
        const int ncon = J.ncon;
        if (ncon == 0) {  // a flat range
            if (x) atomicOr(&J.out[w0 + lane], x);
            continue;
        }
        if (!__any_sync(0xffffffffu, x != 0)) continue;
        kept[lane] = 0;
        const uint32_t n = expand_bits(x, list, lane);
        for (uint32_t i = 0; i < n; i += 32) {
            const bool valid = i + lane < n;
            const uint32_t at = valid ? list[i + lane] : 0u, v = w0 * 32 + at;
            bool keep = valid;
            for (int c = 0; c < ncon; c++) {
                const AdjRef A = adj_ref(g, J.con_dir[c]);
                const int32_t lab = J.con_lab[c];
                const uint32_t* bm = J.con_bm[c];
                uint32_t e0 = 0, e1 = 0;
                if (keep) {
                    e0 = A.off[v];
                    e1 = A.off[v + 1];
                }
                sc += keep;
                bool hit = false;
                if (J.con_any[c] && e0 < e1) {
                    const uint32_t b = e0 & ~3u;
                    uint32_t y[4], w[4];
                    hit = quad_hits(g, A.adj, b, quad_mask(b, e0, e1), lab, bm, y, w) != 0;
                    if (COUNT) se += min(4u - (e0 - b), e1 - e0);
                    e0 = hit || e1 - b <= 4u ? e1 : b + 4;
                }
                se += e1 - e0;
                found[lane] = hit;
                uint32_t total;
                const uint32_t ex = list_starts(e1 - e0, lane, &total);
                scan_flat(g, A, e0, e1 - e0, ex, total, lab, bm, slots, lane,
                          [&](bool h, uint32_t, uint32_t, int owner, uint32_t) {
                              if (h) found[owner] = 1;
                          });
                keep = keep && found[lane];
            }
            if (keep) atomicOr(&kept[at >> 5], 1u << (at & 31));
        }
        __syncwarp();
        if (lane < (int)nw && kept[lane]) atomicOr(&J.out[w0 + lane], kept[lane]);
        __syncwarp();  // list and kept are written again
    }
    scan_flush<COUNT>(scan, sc, se);
}

__global__ void __launch_bounds__(FILTER_THREADS) k_clear(DevGraph g, const RefineJob* __restrict__ jobs, int njobs) {
    for (int j = blockIdx.y; j < njobs; j += gridDim.y)
        for (uint32_t w = blockIdx.x * FILTER_THREADS + threadIdx.x; w < g.nwords; w += gridDim.x * FILTER_THREADS)
            jobs[j].out[w] = 0;
}

// Position in the parent's candidate list of the first candidate at or after
// vertex a.
__device__ __forceinline__ uint32_t parent_rank(const CpiJob& J, uint32_t a) {
    return J.prank[a >> 5] + __popc(J.r.bm[a >> 5] & ((1u << (a & 31)) - 1u));
}

// off[a] = number of children of parent candidate a
template <bool COUNT>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS, SCAN_BLOCKS) k_cpi_count(DevGraph g, const CpiJob* __restrict__ jobs,
                                                                   int njobs, ScanLaunch l, ScanCount scan) {
    using Reduce = cub::BlockReduce<uint32_t, WARP_KERNEL_THREADS>;
    __shared__ typename Reduce::TempStorage tmp;
    __shared__ ScanShared sh;
    const int lane = threadIdx.x & 31;
    int2* const slots = sh.slots + (threadIdx.x & ~31);
    uint16_t* const list = sh.list[threadIdx.x >> 5];
    uint64_t sc = 0, se = 0;
    for (uint32_t it = blockIdx.x; it < l.hubs; it += gridDim.x) {
        uint32_t at;
        const CpiJob& J = jobs[job_of(l.hub_first, njobs, it, &at)];
        const uint32_t v = J.r.lo[0] + at;
        if (!((J.r.bm[v >> 5] >> (v & 31)) & 1u)) continue;
        const AdjRef A = adj_ref(g, J.out);
        const uint32_t e0 = A.off[v], e1 = A.off[v + 1];
        if (threadIdx.x == 0) sc += e1 > e0, se += e1 - e0;
        uint32_t cnt = 0;
        scan_block(g, A.adj, e0, e1, J.lab, J.cbm,
                   [&](int, uint32_t h, const uint32_t (&)[4], const uint32_t (&)[4]) { cnt += __popc(h); },
                   [] { return false; });
        const uint32_t total = Reduce(tmp).Sum(cnt);
        if (threadIdx.x == 0) J.off[parent_rank(J, v)] = total;
        __syncthreads();  // tmp is reused by the next hub
    }
    for (uint64_t it = gwarp_id(); it < l.items; it += nwarps_total()) {
        uint32_t item, va, vb;
        const CpiJob& J = jobs[job_of(l.first, njobs, (uint32_t)it, &item)];
        item_range(J.r, item, l, &va, &vb);
        const uint32_t w0 = va >> 5, nw = (vb + 31) / 32 - w0;
        const uint32_t x = lane < (int)nw ? J.r.bm[w0 + lane] & item_mask(w0 + lane, va, vb) : 0u;
        if (!__any_sync(0xffffffffu, x != 0)) continue;
        const uint32_t n = expand_bits(x, list, lane);
        const AdjRef A = adj_ref(g, J.out);
        uint32_t* const off = J.off + parent_rank(J, va);
        for (uint32_t i = 0; i < n; i += 32) {
            const bool valid = i + lane < n;
            uint32_t e0 = 0, e1 = 0;
            if (valid) {
                const uint32_t v = w0 * 32 + list[i + lane];
                e0 = A.off[v];
                e1 = A.off[v + 1];
            }
            sc += e1 > e0;
            se += e1 - e0;
            uint32_t total, cnt = 0;
            const uint32_t len = e1 - e0, ex = list_starts(len, lane, &total);
            scan_flat(g, A, e0, len, ex, total, J.lab, J.cbm, slots, lane,
                      [&](bool hit, uint32_t, uint32_t, int, uint32_t window) {
                          const uint32_t hits = __ballot_sync(0xffffffffu, hit);
                          // the window's entries of this lane's list: [ex, ex + len)
                          if (hits && len && window + 32u > ex && window < ex + len) {
                              const uint32_t lo = ex > window ? ex - window : 0u;
                              const uint32_t hi = min(ex + len - window, 32u);
                              cnt += __popc((hits >> lo) << (32u - hi + lo));
                          }
                      });
            if (valid) off[i + lane] = cnt;
        }
        __syncwarp();  // list is written again
    }
    scan_flush<COUNT>(scan, sc, se);
}

// Exclusive scan of the per-candidate counts off[0..n) in place, off[n] =
// total, in two passes over the jobs' chunks of CPI_CHUNK counts (as many as the
// parent's label has vertices for) like the compaction above.
__device__ __forceinline__ const CpiJob& chunk_job(const CpiJob* jobs, int njobs, uint32_t it, uint32_t* c) {
    int lo = 0, hi = njobs;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (jobs[mid].chunk0 <= it) lo = mid;
        else hi = mid;
    }
    *c = it - jobs[lo].chunk0;
    return jobs[lo];
}

__global__ void __launch_bounds__(COMPACT_THREADS) k_cpi_sums(const CpiJob* __restrict__ jobs, int njobs,
                                                              uint32_t chunks) {
    using Reduce = cub::BlockReduce<uint64_t, COMPACT_THREADS>;
    __shared__ typename Reduce::TempStorage tmp;
    for (uint32_t it = blockIdx.x; it < chunks; it += gridDim.x) {
        uint32_t c;
        const CpiJob& J = chunk_job(jobs, njobs, it, &c);
        const uint32_t n = *J.pcount;
        if ((uint64_t)c * CPI_CHUNK >= n && c > 0) continue;
        uint64_t cnt = 0;
        for (uint32_t a = c * CPI_CHUNK + threadIdx.x; a < min(n, (c + 1) * CPI_CHUNK); a += COMPACT_THREADS)
            cnt += J.off[a];
        cnt = Reduce(tmp).Sum(cnt);
        if (threadIdx.x == 0) J.csum[c] = cnt;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(COMPACT_THREADS) k_cpi_scan(const CpiJob* __restrict__ jobs, int njobs,
                                                              uint32_t chunks, int32_t* err) {
    using Scan = cub::BlockScan<uint64_t, COMPACT_THREADS>;
    using Reduce = cub::BlockReduce<uint64_t, COMPACT_THREADS>;
    __shared__ union {
        typename Scan::TempStorage scan;
        typename Reduce::TempStorage reduce;
    } tmp;
    __shared__ uint64_t base_s;
    constexpr int EPT = CPI_CHUNK / COMPACT_THREADS;
    for (uint32_t it = blockIdx.x; it < chunks; it += gridDim.x) {
        uint32_t c;
        const CpiJob& J = chunk_job(jobs, njobs, it, &c);
        const uint32_t n = *J.pcount;
        const uint32_t last = n / CPI_CHUNK;  // chunk holding off[n]
        if (c > last) continue;
        uint64_t before = 0;
        for (uint32_t q = threadIdx.x; q < c; q += COMPACT_THREADS) before += J.csum[q];
        before = Reduce(tmp.reduce).Sum(before);
        if (threadIdx.x == 0) base_s = before;
        __syncthreads();
        const uint32_t a0 = c * CPI_CHUNK + threadIdx.x * EPT;
        uint32_t vals[EPT];
        uint64_t cnt = 0;
        for (int q = 0; q < EPT; q++) {
            vals[q] = a0 + q < n ? J.off[a0 + q] : 0u;
            cnt += vals[q];
        }
        uint64_t excl, total;
        Scan(tmp.scan).ExclusiveSum(cnt, excl, total);
        uint64_t r = base_s + excl;
        const bool overflow = base_s + total > J.cap || base_s + total > 0xffffffffull;
        for (int q = 0; q < EPT; q++) {
            if (a0 + q >= n) break;
            J.off[a0 + q] = overflow ? 0u : (uint32_t)r;
            r += vals[q];
        }
        if (c == last && threadIdx.x == 0) {
            uint64_t tot = base_s + total;
            if (overflow) {
                atomicExch(err, DERR_CAPACITY);
                tot = 0;  // leave an empty index
            }
            J.off[n] = (uint32_t)tot;
            *J.total = (uint32_t)tot;
        }
        __syncthreads();
    }
}

// Index edges of an item's parents are contiguous and in scan order, so the
// warp only counts hits. A hub's edges are put in order by a block scan of the
// threads' hits (HUB_QUADS quads in a row each) per round.
template <bool COUNT>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS, SCAN_BLOCKS) k_cpi_fill(DevGraph g, const CpiJob* __restrict__ jobs, int njobs,
                                                                  ScanLaunch l, ScanCount scan) {
    using Scan = cub::BlockScan<uint32_t, WARP_KERNEL_THREADS>;
    __shared__ typename Scan::TempStorage tmp;
    __shared__ ScanShared sh;
    const int lane = threadIdx.x & 31;
    int2* const slots = sh.slots + (threadIdx.x & ~31);
    uint16_t* const list = sh.list[threadIdx.x >> 5];
    uint64_t sc = 0, se = 0;
    for (uint32_t it = blockIdx.x; it < l.hubs; it += gridDim.x) {
        uint32_t at;
        const CpiJob& J = jobs[job_of(l.hub_first, njobs, it, &at)];
        const uint32_t v = J.r.lo[0] + at;
        if (!((J.r.bm[v >> 5] >> (v & 31)) & 1u)) continue;
        const uint32_t a = parent_rank(J, v);
        uint32_t next = J.off[a];
        const uint32_t end = J.off[a + 1];
        if (next == end) continue;  // no index edges
        const AdjRef A = adj_ref(g, J.out);
        const uint32_t e0 = A.off[v], e1 = A.off[v + 1];
        if (threadIdx.x == 0) sc += 1, se += e1 - e0;
        uint32_t hq[HUB_QUADS] = {}, xq[HUB_QUADS][4];
        scan_block(g, A.adj, e0, e1, J.lab, J.cbm,
                   [&](int q, uint32_t h, const uint32_t (&x)[4], const uint32_t (&)[4]) {
#pragma unroll
                       for (int i = 0; i < HUB_QUADS; i++)
                           if (i == q) {
                               hq[i] = h;
#pragma unroll
                               for (int c = 0; c < 4; c++) xq[i][c] = x[c];
                           }
                   },
                   [&] {
                       uint32_t mine = 0, excl, total;
#pragma unroll
                       for (int i = 0; i < HUB_QUADS; i++) mine += __popc(hq[i]);
                       Scan(tmp).ExclusiveSum(mine, excl, total);
                       uint32_t slot = next + excl;
#pragma unroll
                       for (int i = 0; i < HUB_QUADS; i++) {
#pragma unroll
                           for (int c = 0; c < 4; c++)
                               if ((hq[i] >> c) & 1u) {
                                   const uint32_t x = xq[i][c];
                                   if (slot < J.cap && J.ids)
                                       reinterpret_cast<uint32_t*>(J.idx)[slot] = x;
                                   else if (slot < J.cap)
                                       J.idx[slot] = make_int2((int32_t)(__ldg(J.crank + (x >> 5)) +
                                                                         __popc(__ldg(J.cbm + (x >> 5)) &
                                                                                ((1u << (x & 31)) - 1))), (int32_t)x);
                                   slot++;
                               }
                           hq[i] = 0;
                       }
                       next += total;
                       __syncthreads();  // tmp is reused by the next round
                       return next >= end;
                   });
    }
    for (uint64_t it = gwarp_id(); it < l.items; it += nwarps_total()) {
        uint32_t item, va, vb;
        const CpiJob& J = jobs[job_of(l.first, njobs, (uint32_t)it, &item)];
        item_range(J.r, item, l, &va, &vb);
        const uint32_t w0 = va >> 5, nw = (vb + 31) / 32 - w0;
        const uint32_t x = lane < (int)nw ? J.r.bm[w0 + lane] & item_mask(w0 + lane, va, vb) : 0u;
        if (!__any_sync(0xffffffffu, x != 0)) continue;
        const uint32_t n = expand_bits(x, list, lane);
        const AdjRef A = adj_ref(g, J.out);
        const uint32_t* const off = J.off + parent_rank(J, va);
        int2* const idx = J.idx;
        const bool ids = J.ids;
        const uint32_t* const crank = J.crank;
        const uint64_t cap = J.cap;
        for (uint32_t i = 0; i < n; i += 32) {
            uint32_t e0 = 0, e1 = 0, o = 0;
            if (i + lane < n) {
                o = off[i + lane];
                if (off[i + lane + 1] > o) {  // a parent without index edges skips its list
                    const uint32_t v = w0 * 32 + list[i + lane];
                    e0 = A.off[v];
                    e1 = A.off[v + 1];
                }
            }
            sc += e1 > e0;
            se += e1 - e0;
            uint32_t total;
            const uint32_t ex = list_starts(e1 - e0, lane, &total);
            uint32_t next = __shfl_sync(0xffffffffu, o, 0);
            scan_flat(g, A, e0, e1 - e0, ex, total, J.lab, J.cbm, slots, lane,
                      [&](bool hit, uint32_t y, uint32_t w, int, uint32_t) {
                          const uint32_t hits = __ballot_sync(0xffffffffu, hit);
                          if (hit) {
                              const uint32_t slot = next + __popc(hits & ((1u << lane) - 1u));
                              if (slot < cap && ids)
                                  reinterpret_cast<uint32_t*>(idx)[slot] = y;
                              else if (slot < cap)
                                  idx[slot] = make_int2((int32_t)(__ldg(crank + (y >> 5)) +
                                                                  __popc(w & ((1u << (y & 31)) - 1))), (int32_t)y);
                          }
                          next += __popc(hits);
                      });
        }
        __syncwarp();  // list is written again
    }
    scan_flush<COUNT>(scan, sc, se);
}

// Blocks of a grid-stride kernel: as many as the device holds at once. A
// larger grid leaves a partial second wave, whose blocks start only as
// first-wave blocks exit and then run their share at a fraction of the
// occupancy. Cached per (kernel, device).
int resident_grid(const void* fn, int threads) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    const int sms = device_sms();
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(fn, dev);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, 0) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();  // the launch itself reports a kernel that cannot run
        per_sm = 1;
    }
    const int grid = sms * per_sm;
    cache.emplace(key, grid);
    return grid;
}

template <typename F>
int grid_of(F* fn, int threads) {
    return resident_grid((const void*)fn, threads);
}

int check_launch(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, what);
    return GFD_OK;
}

}  // namespace

int launch_filter(const DevGraph& g, const FilterKey* d_keys, int nkeys, uint32_t* d_out, cudaStream_t st) {
    if (nkeys <= 0 || g.nwords == 0) return GFD_OK;
    int blocks = (int)std::min<uint64_t>((g.nwords * 32 + FILTER_THREADS - 1) / FILTER_THREADS, (uint64_t)device_sms() * 8);
    // keys staged in shared memory: at most KEYS_PER_LAUNCH per launch
    constexpr int KEYS_PER_LAUNCH = 4096;
    for (int k0 = 0; k0 < nkeys; k0 += KEYS_PER_LAUNCH) {
        const int cnt = std::min(KEYS_PER_LAUNCH, nkeys - k0);
        const size_t smem = sizeof(FilterKey) * cnt;
        if (smem > 48 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(k_filter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(k_filter)");
        }
        k_filter<<<std::max(blocks, 1), FILTER_THREADS, smem, st>>>(g, d_keys + k0, cnt,
                                                                    d_out + (uint64_t)k0 * g.nwords);
        if (int rc = check_launch("k_filter")) return rc;
    }
    return GFD_OK;
}

int launch_clear(const DevGraph& g, const RefineJob* d_jobs, int njobs, cudaStream_t st) {
    if (njobs <= 0 || g.nwords == 0) return GFD_OK;
    const uint32_t wide = std::min<uint32_t>((g.nwords + FILTER_THREADS - 1) / FILTER_THREADS, 64);
    k_clear<<<dim3(wide, (unsigned)std::min(njobs, 1024)), FILTER_THREADS, 0, st>>>(g, d_jobs, njobs);
    return check_launch("k_clear");
}

uint32_t compact_chunks(const DevGraph& g) {
    return std::max<uint32_t>(1, (g.nwords + COMPACT_WORDS - 1) / COMPACT_WORDS);
}

int launch_compact(const DevGraph& g, const CompactJob* d_jobs, int njobs, cudaStream_t st) {
    if (njobs <= 0) return GFD_OK;
    const uint32_t nch = compact_chunks(g);
    const int grid = (int)std::min<uint64_t>((uint64_t)njobs * nch, (uint64_t)device_sms() * 8);
    k_compact_sums<<<grid, COMPACT_THREADS, 0, st>>>(g, d_jobs, njobs, nch);
    k_compact_write<<<grid, COMPACT_THREADS, 0, st>>>(g, d_jobs, njobs, nch);
    return check_launch("k_compact");
}

uint32_t cpi_chunks(uint64_t max_parent_candidates) { return (uint32_t)(max_parent_candidates / CPI_CHUNK + 1); }

// A large launch takes larger units, so that its warps' lanes fill up although the
// bitmaps are sparse and an item's fixed cost (finding its job, its words) is
// spread; a small one smaller units, so that its few candidates reach all SMs and
// no warp gets more than 2048 entries at a time. In between, the last class's unit leaves
// every resident warp about four items, up to 2^most vertices: 8 for refinement,
// whose bitmaps are dense at first (batch of 256 GFDs on 4M vertices: 55 / 48 / 44 /
// 38 / 38.5 ms at 5 .. 9, with units of 4 to 8 vertices in class 1 and 32 to 64 in
// class 2 from 8 on; 45 ms with 32 in class 1, whose warps then get 64k entries),
// 10 for the index edges, whose parents are sparse (23.9 / 21.9 / 21.7 ms at 8 ..
// 10; 43.6 ms with units of 128 vertices in the last class and 8 in class 2).
void scan_units(uint64_t vertices, int most, int8_t* unit) {
    const uint64_t per_warp = vertices / ((uint64_t)device_sms() * 48 * 4);
    int u = 5;
    while (u < most && (2ull << u) <= per_warp) u++;
    unit[0] = 0;
    unit[1] = u >= 8 ? 2 : 0;
    unit[2] = u >= 8 ? 6 : 3;
    unit[3] = (int8_t)u;
}

namespace {

// At most one resident wave, at least a warp per item and a block per hub.
template <typename Job>
int launch_scan(void (*kernel)(DevGraph, const Job*, int, ScanLaunch, ScanCount), const DevGraph& g, const Job* d_jobs,
                int njobs, const ScanLaunch& l, ScanCount scan, cudaStream_t st, const char* what) {
    const uint64_t want = std::max<uint64_t>(((uint64_t)l.items + WARP_KERNEL_THREADS / 32 - 1) / (WARP_KERNEL_THREADS / 32), l.hubs);
    if (njobs <= 0 || want == 0) return GFD_OK;
    const int grid = (int)std::min<uint64_t>(want, (uint64_t)grid_of(kernel, WARP_KERNEL_THREADS));
    kernel<<<grid, WARP_KERNEL_THREADS, 0, st>>>(g, d_jobs, njobs, l, scan);
    return check_launch(what);
}

}  // namespace

int launch_scatter(const DevGraph& g, const ScatterJob* d_jobs, int njobs, const ScanLaunch& l, ScanCount scan,
                   cudaStream_t st) {
    return launch_scan(scan ? k_scatter<true> : k_scatter<false>, g, d_jobs, njobs, l, scan, st, "k_scatter");
}

int launch_refine(const DevGraph& g, const RefineJob* d_jobs, int njobs, const ScanLaunch& l, ScanCount scan,
                  cudaStream_t st) {
    return launch_scan(scan ? k_refine<true> : k_refine<false>, g, d_jobs, njobs, l, scan, st, "k_refine");
}

int launch_cpi_count(const DevGraph& g, const CpiJob* d_jobs, int njobs, const ScanLaunch& l, uint32_t chunks,
                     int32_t* d_err, ScanCount scan, cudaStream_t st) {
    if (njobs <= 0) return GFD_OK;
    if (int rc = launch_scan(scan ? k_cpi_count<true> : k_cpi_count<false>, g, d_jobs, njobs, l, scan, st, "k_cpi_count"))
        return rc;
    const int grid = (int)std::min<uint64_t>(chunks, (uint64_t)device_sms() * 8);
    k_cpi_sums<<<grid, COMPACT_THREADS, 0, st>>>(d_jobs, njobs, chunks);
    k_cpi_scan<<<grid, COMPACT_THREADS, 0, st>>>(d_jobs, njobs, chunks, d_err);
    return check_launch("k_cpi_scan");
}

int launch_cpi_fill(const DevGraph& g, const CpiJob* d_jobs, int njobs, const ScanLaunch& l, ScanCount scan,
                    cudaStream_t st) {
    return launch_scan(scan ? k_cpi_fill<true> : k_cpi_fill<false>, g, d_jobs, njobs, l, scan, st, "k_cpi_fill");
}

}  // namespace gfd
