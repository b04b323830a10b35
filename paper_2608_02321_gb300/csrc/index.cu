// Compact path index construction (Section III.B, step 1).
//
//   k_filter   step 1a-1b: candidates by label and degree (and self-loop, and
//              pushed-down constant X literals), one coalesced pass over vertex
//              data for all filter keys;
//   k_scatter  step 1c: mark vertices adjacent (in the direction and with the
//   k_and      label of a pattern edge) to the candidates of another level,
//              then intersect;
//   k_prune    step 1c: remove candidates with no such neighbour among the
//              candidates of another level (early exit at the first one);
//              top-down and bottom-up use whichever of the two is cheaper;
//   k_compact  bitmap -> exclusive popcount prefix (O(1) rank) + sorted list;
//   k_cpi_*    step 1d: for each spanning-tree edge, the index edges from
//              every parent candidate to the positions of its child candidates;
// The adjacency scans (k_scatter, k_prune, k_cpi_count, k_cpi_fill) share out a
// job's candidates by degree class: a block per hub, a warp per 1, 8 or 32
// vertices of the other classes.
//
// Every launch processes a table of jobs; blocks (or warps) stride over the
// items of each job with a per-job rotation so that small jobs spread out.
#include <cub/cub.cuh>

#include <algorithm>
#include <map>
#include <mutex>

#include "engine.h"

namespace gfd {

namespace {

constexpr int FILTER_THREADS = 256;
constexpr int COMPACT_THREADS = 256;
constexpr uint32_t COMPACT_WORDS = 1024;  // words (or counts) per chunk
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

// One block per (job, chunk of AND_WORDS words) item, so that every job's words
// are spread over the GPU and no thread walks the job table.
constexpr uint32_t AND_WORDS = 2048;
constexpr int AND_THREADS = 256;

__global__ void __launch_bounds__(AND_THREADS) k_and(DevGraph g, const AndJob* __restrict__ jobs, int njobs,
                                                      uint32_t nchunks) {
    for (uint64_t it = blockIdx.x; it < (uint64_t)njobs * nchunks; it += gridDim.x) {
        const AndJob& J = jobs[it / nchunks];
        const uint32_t w0 = (uint32_t)(it % nchunks) * AND_WORDS;
        const uint32_t w1 = min(g.nwords, w0 + AND_WORDS);
        const int ntmp = J.ntmp;
        for (uint32_t w = w0 + threadIdx.x; w < w1; w += AND_THREADS) {
            uint32_t x = J.src[w];
            for (int t = 0; t < ntmp; t++) x &= J.tmp[t][w];
            J.bm[w] = x;
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
        for (int q = 0; q < WPT; q++)
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

// The adjacency kernels below give the lanes of a warp a candidate each (32 of
// the lowest degree class, fewer of the others); the warp then scans its lists
// end to end as one sequence, 32 x FLAT entries at a time (scan_flat). A hub's
// list is scanned by a block. Vertices are numbered by degree class, so a
// candidate list holds its classes one after the other, and where they end are
// rank lookups.
//
// These scans are bound by latency (a random adjacency line, then a random
// bitmap word, from L2 or HBM) and by balance. A lane that scans its own list
// leaves the warp waiting for its longest list with few loads in flight; a warp
// that happens to get 32 long lists keeps the launch waiting. End to end every
// lane has FLAT loads in flight whatever the degrees, and by classes no warp
// gets more than 2048 entries at a time.
constexpr int FLAT = 4;
// candidates per warp of each class after the hubs (x the class's largest degree:
// at most 2048 entries)
__device__ constexpr uint32_t class_group(int c) { return c == 1 ? 1 : c == 2 ? 8 : 32; }

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

// Work of a launch over all its jobs, written by k_job_groups: ScanWork::pre
// holds, for the J = njobs jobs, the exclusive prefix of their warp groups
// [J + 1], that of their hubs [J + 1], and per job where its first classes end in
// the candidate list [(N_CLASS - 1) J]. Groups and hubs are taken from one flat
// index each; job_of finds an item's job by binary search.
__device__ __forceinline__ const ScanList& list_of(const ScatterJob& J) { return J.q; }
__device__ __forceinline__ const ScanList& list_of(const PruneJob& J) { return J.c; }
__device__ __forceinline__ const ScanList& list_of(const CpiJob& J) { return J.p; }

constexpr int JOB_SCAN_THREADS = 1024;

// candidates of the list below vertex v (its bitmap and ranks as compacted)
__device__ __forceinline__ uint32_t list_rank(const DevGraph& g, const ScanList& C, uint32_t v) {
    if (v >= (uint32_t)g.n) return *C.count;
    return C.rank[v >> 5] + __popc(C.bm[v >> 5] & ((1u << (v & 31)) - 1u));
}

template <typename Job>
__global__ void __launch_bounds__(JOB_SCAN_THREADS) k_job_groups(DevGraph g, const Job* __restrict__ jobs, int njobs,
                                                                  uint32_t* pre) {
    using Scan = cub::BlockScan<uint32_t, JOB_SCAN_THREADS>;
    __shared__ typename Scan::TempStorage tmp;
    __shared__ uint32_t carry[2];
    uint32_t* const hpre = pre + njobs + 1;
    uint32_t* const cls = hpre + njobs + 1;
    if (threadIdx.x < 2) carry[threadIdx.x] = 0;
    __syncthreads();
    for (int b = 0; b < njobs; b += JOB_SCAN_THREADS) {
        const int j = b + threadIdx.x;
        uint32_t groups = 0, hubs = 0;
        if (j < njobs) {
            const ScanList& C = list_of(jobs[j]);
            uint32_t begin = hubs = list_rank(g, C, g.class_end[0]);
            cls[(N_CLASS - 1) * j] = hubs;
            for (int c = 1; c < N_CLASS; c++) {
                const uint32_t end = c < N_CLASS - 1 ? list_rank(g, C, g.class_end[c]) : *C.count;
                if (c < N_CLASS - 1) cls[(N_CLASS - 1) * j + c] = end;
                groups += (end - begin + class_group(c) - 1) / class_group(c);
                begin = end;
            }
        }
        uint32_t excl, total, hexcl, htotal;
        Scan(tmp).ExclusiveSum(groups, excl, total);
        __syncthreads();
        Scan(tmp).ExclusiveSum(hubs, hexcl, htotal);
        if (j < njobs) {
            pre[j] = carry[0] + excl;
            hpre[j] = carry[1] + hexcl;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            carry[0] += total;
            carry[1] += htotal;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        pre[njobs] = carry[0];
        hpre[njobs] = carry[1];
    }
}

// the job whose items [pre[j], pre[j+1]) hold item it (pre[njobs] > it)
__device__ __forceinline__ int job_of(const uint32_t* pre, int njobs, uint32_t it) {
    int lo = 0, hi = njobs;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(pre + mid) <= it) lo = mid;
        else hi = mid;
    }
    return lo;
}

// A launch's hubs (item = job, position in its candidate list) and warp groups.
struct Groups {
    const uint32_t *pre, *hpre, *cls;
    int njobs;
    __device__ __forceinline__ Groups(const ScanWork& w, int n)
        : pre(w.pre), hpre(w.pre + n + 1), cls(w.pre + 2 * (n + 1)), njobs(n) {}
    __device__ __forceinline__ uint32_t n_groups() const { return pre[njobs]; }
    __device__ __forceinline__ uint32_t n_hubs() const { return hpre[njobs]; }
    __device__ __forceinline__ int hub(uint32_t it, uint32_t* a) const {
        const int j = job_of(hpre, njobs, it);
        *a = it - hpre[j];
        return j;
    }
    // job of group it; a: the lane's position in its candidate list (from the
    // list's end on for a lane without a candidate)
    __device__ __forceinline__ int group(uint32_t it, uint32_t lane, uint32_t* a) const {
        const int j = job_of(pre, njobs, it);
        const uint32_t* const end = cls + (N_CLASS - 1) * j;
        uint32_t grp = it - pre[j], begin = end[0];
#pragma unroll
        for (int c = 1; c < N_CLASS - 1; c++) {
            const uint32_t groups = (end[c] - begin + class_group(c) - 1) / class_group(c);
            if (grp < groups) {
                begin += grp * class_group(c) + lane;
                *a = lane < class_group(c) && begin < end[c] ? begin : 0xffffffffu;
                return j;
            }
            grp -= groups;
            begin = end[c];
        }
        *a = begin + grp * 32 + lane;
        return j;
    }
};

// Counting pass: add this thread's scanned candidates and adjacency entries to
// the run's counters (all lanes of the warp call it; one atomic per warp).
template <bool COUNT>
__device__ __forceinline__ void scan_flush(const ScanWork& q, uint64_t cands, uint64_t entries) {
    if (!COUNT || !q.scan) return;
    for (int d = 16; d >= 1; d >>= 1) {
        cands += __shfl_xor_sync(0xffffffffu, cands, d);
        entries += __shfl_xor_sync(0xffffffffu, entries, d);
    }
    if ((threadIdx.x & 31) == 0) {
        if (cands) atomicAdd(&q.scan[0], (unsigned long long)cands);
        if (entries) atomicAdd(&q.scan[1], (unsigned long long)entries);
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

template <bool COUNT>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS) k_scatter(DevGraph g, const ScatterJob* __restrict__ jobs,
                                                                 int njobs, ScanWork sw) {
    __shared__ int2 s_slots[WARP_KERNEL_THREADS];
    const int lane = threadIdx.x & 31;
    int2* const slots = s_slots + (threadIdx.x & ~31);
    const Groups G(sw, njobs);
    uint64_t sc = 0, se = 0;
    const uint32_t nhubs = G.n_hubs();
    for (uint32_t it = blockIdx.x; it < nhubs; it += gridDim.x) {
        uint32_t a;
        const ScatterJob& J = jobs[G.hub(it, &a)];
        const AdjRef A = adj_ref(g, J.scan_out);
        const uint32_t v = (uint32_t)J.q.cand[a], e0 = A.off[v], e1 = A.off[v + 1];
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
    const uint32_t ngroups = G.n_groups();
    for (uint64_t it = gwarp_id(); it < ngroups; it += nwarps_total()) {
        uint32_t a;
        const ScatterJob& J = jobs[G.group((uint32_t)it, lane, &a)];
        const AdjRef A = adj_ref(g, J.scan_out);
        uint32_t e0 = 0, e1 = 0;
        if (a < *J.q.count) {
            const uint32_t v = (uint32_t)J.q.cand[a];
            e0 = A.off[v];
            e1 = A.off[v + 1];
        }
        sc += e1 > e0;
        se += e1 - e0;
        uint32_t total;
        const uint32_t ex = list_starts(e1 - e0, lane, &total);
        uint32_t* const marks = J.marks;
        scan_flat(g, A, e0, e1 - e0, ex, total, J.lab, J.filter, slots, lane,
                  [&](bool hit, uint32_t x, uint32_t, int, uint32_t) {
                      if (hit) mark(marks, x);
                  });
    }
    scan_flush<COUNT>(sw, sc, se);
}

// A constraint on neighbours of any vertex label hits often: each lane first
// tries its own list's first quad, and only lists without a hit there are
// scanned end to end.
template <bool COUNT>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS) k_prune(DevGraph g, const PruneJob* __restrict__ jobs, int njobs,
                                                               ScanWork sw) {
    __shared__ int2 s_slots[WARP_KERNEL_THREADS];
    __shared__ uint8_t s_hit[WARP_KERNEL_THREADS];
    const int lane = threadIdx.x & 31;
    int2* const slots = s_slots + (threadIdx.x & ~31);
    uint8_t* const found = s_hit + (threadIdx.x & ~31);
    const Groups G(sw, njobs);
    uint64_t sc = 0, se = 0;
    const uint32_t nhubs = G.n_hubs();
    for (uint32_t it = blockIdx.x; it < nhubs; it += gridDim.x) {
        uint32_t a;
        const PruneJob& J = jobs[G.hub(it, &a)];
        const uint32_t v = (uint32_t)J.c.cand[a];
        bool keep = true;
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
        if (!keep && threadIdx.x == 0) atomicAnd(&J.out[v >> 5], ~(1u << (v & 31)));
    }
    const uint32_t ngroups = G.n_groups();
    for (uint64_t it = gwarp_id(); it < ngroups; it += nwarps_total()) {
        uint32_t a;
        const PruneJob& J = jobs[G.group((uint32_t)it, lane, &a)];
        const int ncon = J.ncon;
        const bool valid = a < *J.c.count;
        const uint32_t v = valid ? (uint32_t)J.c.cand[a] : 0u;
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
                uint32_t x[4], w[4];
                hit = quad_hits(g, A.adj, b, quad_mask(b, e0, e1), lab, bm, x, w) != 0;
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
        if (valid && !keep) atomicAnd(&J.out[v >> 5], ~(1u << (v & 31)));
    }
    scan_flush<COUNT>(sw, sc, se);
}

// off[a] = number of children of parent candidate a
template <bool COUNT>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS) k_cpi_count(DevGraph g, const CpiJob* __restrict__ jobs,
                                                                   int njobs, ScanWork sw) {
    using Reduce = cub::BlockReduce<uint32_t, WARP_KERNEL_THREADS>;
    __shared__ typename Reduce::TempStorage tmp;
    __shared__ int2 s_slots[WARP_KERNEL_THREADS];
    const int lane = threadIdx.x & 31;
    int2* const slots = s_slots + (threadIdx.x & ~31);
    const Groups G(sw, njobs);
    uint64_t sc = 0, se = 0;
    const uint32_t nhubs = G.n_hubs();
    for (uint32_t it = blockIdx.x; it < nhubs; it += gridDim.x) {
        uint32_t a;
        const CpiJob& J = jobs[G.hub(it, &a)];
        const AdjRef A = adj_ref(g, J.out);
        const uint32_t v = (uint32_t)J.p.cand[a], e0 = A.off[v], e1 = A.off[v + 1];
        if (threadIdx.x == 0) sc += e1 > e0, se += e1 - e0;
        uint32_t cnt = 0;
        scan_block(g, A.adj, e0, e1, J.lab, J.cbm,
                   [&](int, uint32_t h, const uint32_t (&)[4], const uint32_t (&)[4]) { cnt += __popc(h); },
                   [] { return false; });
        const uint32_t total = Reduce(tmp).Sum(cnt);
        if (threadIdx.x == 0) J.off[a] = total;
        __syncthreads();  // tmp is reused by the next hub
    }
    const uint32_t ngroups = G.n_groups();
    for (uint64_t it = gwarp_id(); it < ngroups; it += nwarps_total()) {
        uint32_t a;
        const CpiJob& J = jobs[G.group((uint32_t)it, lane, &a)];
        const AdjRef A = adj_ref(g, J.out);
        const bool valid = a < *J.p.count;
        uint32_t e0 = 0, e1 = 0;
        if (valid) {
            const uint32_t v = (uint32_t)J.p.cand[a];
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
        if (valid) J.off[a] = cnt;
    }
    scan_flush<COUNT>(sw, sc, se);
}

// Exclusive scan of the per-candidate counts off[0..n) in place, off[n] =
// total, in two passes over (job, chunk) items like the compaction above.
__global__ void __launch_bounds__(COMPACT_THREADS) k_cpi_sums(const CpiJob* __restrict__ jobs, int njobs,
                                                              uint32_t nchunks) {
    using Reduce = cub::BlockReduce<uint64_t, COMPACT_THREADS>;
    __shared__ typename Reduce::TempStorage tmp;
    for (uint64_t it = blockIdx.x; it < (uint64_t)njobs * nchunks; it += gridDim.x) {
        const CpiJob& J = jobs[it / nchunks];
        const uint32_t c = (uint32_t)(it % nchunks);
        const uint32_t n = *J.p.count;
        if ((uint64_t)c * COMPACT_WORDS >= n && c > 0) continue;
        uint64_t cnt = 0;
        for (uint32_t a = c * COMPACT_WORDS + threadIdx.x; a < min(n, (c + 1) * COMPACT_WORDS); a += COMPACT_THREADS)
            cnt += J.off[a];
        cnt = Reduce(tmp).Sum(cnt);
        if (threadIdx.x == 0) J.csum[c] = cnt;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(COMPACT_THREADS) k_cpi_scan(const CpiJob* __restrict__ jobs, int njobs,
                                                              uint32_t nchunks, int32_t* err) {
    using Scan = cub::BlockScan<uint64_t, COMPACT_THREADS>;
    using Reduce = cub::BlockReduce<uint64_t, COMPACT_THREADS>;
    __shared__ union {
        typename Scan::TempStorage scan;
        typename Reduce::TempStorage reduce;
    } tmp;
    __shared__ uint64_t base_s;
    constexpr int EPT = COMPACT_WORDS / COMPACT_THREADS;
    for (uint64_t it = blockIdx.x; it < (uint64_t)njobs * nchunks; it += gridDim.x) {
        const CpiJob& J = jobs[it / nchunks];
        const uint32_t c = (uint32_t)(it % nchunks);
        const uint32_t n = *J.p.count;
        const uint32_t last = n / COMPACT_WORDS;  // chunk holding off[n]
        if (c > last) continue;
        uint64_t before = 0;
        for (uint32_t q = threadIdx.x; q < c; q += COMPACT_THREADS) before += J.csum[q];
        before = Reduce(tmp.reduce).Sum(before);
        if (threadIdx.x == 0) base_s = before;
        __syncthreads();
        const uint32_t a0 = c * COMPACT_WORDS + threadIdx.x * EPT;
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
            if (J.nnz_stat) atomicAdd((unsigned long long*)J.nnz_stat, (unsigned long long)tot);
        }
        __syncthreads();
    }
}

// Index edges of a group's parents are contiguous and in scan order, so the
// warp only counts hits. A hub's edges are put in order by a block scan of the
// threads' hits (HUB_QUADS quads in a row each) per round.
template <bool COUNT>
__global__ void __launch_bounds__(WARP_KERNEL_THREADS) k_cpi_fill(DevGraph g, const CpiJob* __restrict__ jobs, int njobs,
                                                                  ScanWork sw) {
    using Scan = cub::BlockScan<uint32_t, WARP_KERNEL_THREADS>;
    __shared__ typename Scan::TempStorage tmp;
    __shared__ int2 s_slots[WARP_KERNEL_THREADS];
    const int lane = threadIdx.x & 31;
    int2* const slots = s_slots + (threadIdx.x & ~31);
    const Groups G(sw, njobs);
    uint64_t sc = 0, se = 0;
    const uint32_t nhubs = G.n_hubs();
    for (uint32_t it = blockIdx.x; it < nhubs; it += gridDim.x) {
        uint32_t a;
        const CpiJob& J = jobs[G.hub(it, &a)];
        const AdjRef A = adj_ref(g, J.out);
        const uint32_t v = (uint32_t)J.p.cand[a], e0 = A.off[v], e1 = A.off[v + 1];
        uint32_t next = J.off[a];
        const uint32_t end = J.off[a + 1];
        if (next == end) continue;  // no index edges
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
                                   if (slot < J.cap)
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
    const uint32_t ngroups = G.n_groups();
    for (uint64_t it = gwarp_id(); it < ngroups; it += nwarps_total()) {
        uint32_t a;
        const CpiJob& J = jobs[G.group((uint32_t)it, lane, &a)];
        const AdjRef A = adj_ref(g, J.out);
        uint32_t e0 = 0, e1 = 0, o = 0;
        if (a < *J.p.count) {
            o = J.off[a];
            if (J.off[a + 1] > o) {  // a parent without index edges skips its list
                const uint32_t v = (uint32_t)J.p.cand[a];
                e0 = A.off[v];
                e1 = A.off[v + 1];
            }
        }
        sc += e1 > e0;
        se += e1 - e0;
        uint32_t total;
        const uint32_t ex = list_starts(e1 - e0, lane, &total);
        uint32_t next = __shfl_sync(0xffffffffu, o, 0);
        int2* const idx = J.idx;
        const uint32_t* const crank = J.crank;
        const uint64_t cap = J.cap;
        scan_flat(g, A, e0, e1 - e0, ex, total, J.lab, J.cbm, slots, lane,
                  [&](bool hit, uint32_t x, uint32_t w, int, uint32_t) {
                      const uint32_t hits = __ballot_sync(0xffffffffu, hit);
                      if (hit) {
                          const uint32_t slot = next + __popc(hits & ((1u << lane) - 1u));
                          if (slot < cap)
                              idx[slot] = make_int2((int32_t)(__ldg(crank + (x >> 5)) +
                                                              __popc(w & ((1u << (x & 31)) - 1))), (int32_t)x);
                      }
                      next += __popc(hits);
                  });
    }
    scan_flush<COUNT>(sw, sc, se);
}

// number of index edges of each job (read back to size the index exactly)
__global__ void k_cpi_totals(const CpiJob* __restrict__ jobs, int njobs, uint32_t* totals) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < njobs) totals[j] = jobs[j].off[*jobs[j].p.count];
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

int launch_and(const DevGraph& g, const AndJob* d_jobs, int njobs, cudaStream_t st) {
    if (njobs <= 0 || g.nwords == 0) return GFD_OK;
    const uint32_t nch = (g.nwords + AND_WORDS - 1) / AND_WORDS;
    const int grid = (int)std::min<uint64_t>((uint64_t)njobs * nch, (uint64_t)device_sms() * 16);
    k_and<<<grid, AND_THREADS, 0, st>>>(g, d_jobs, njobs, nch);
    return check_launch("k_and");
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

// the work of a launch over njobs jobs, then the kernel, one resident wave
template <typename Job>
static void job_groups(const DevGraph& g, const Job* d_jobs, int njobs, const ScanWork& sw, cudaStream_t st) {
    k_job_groups<Job><<<1, JOB_SCAN_THREADS, 0, st>>>(g, d_jobs, njobs, sw.pre);
}

#define GFD_SCAN_LAUNCH(kernel)                                                                                   \
    do {                                                                                                          \
        job_groups(g, d_jobs, njobs, sw, st);                                                                     \
        if (sw.scan)                                                                                              \
            kernel<true><<<grid_of(kernel<true>, WARP_KERNEL_THREADS), WARP_KERNEL_THREADS, 0, st>>>(g, d_jobs, njobs, sw); \
        else                                                                                                      \
            kernel<false><<<grid_of(kernel<false>, WARP_KERNEL_THREADS), WARP_KERNEL_THREADS, 0, st>>>(g, d_jobs, njobs, sw); \
    } while (0)

int launch_scatter(const DevGraph& g, const ScatterJob* d_jobs, int njobs, const ScanWork& sw, cudaStream_t st) {
    if (njobs <= 0) return GFD_OK;
    GFD_SCAN_LAUNCH(k_scatter);
    return check_launch("k_scatter");
}

int launch_prune(const DevGraph& g, const PruneJob* d_jobs, int njobs, const ScanWork& sw, cudaStream_t st) {
    if (njobs <= 0) return GFD_OK;
    GFD_SCAN_LAUNCH(k_prune);
    return check_launch("k_prune");
}

uint32_t cpi_chunks(uint64_t max_parent_candidates) {
    return (uint32_t)(max_parent_candidates / COMPACT_WORDS + 1);
}

int launch_cpi_count(const DevGraph& g, const CpiJob* d_jobs, int njobs, uint32_t nchunks, int32_t* d_err,
                     uint32_t* d_totals, const ScanWork& sw, cudaStream_t st) {
    if (njobs <= 0) return GFD_OK;
    GFD_SCAN_LAUNCH(k_cpi_count);
    const int grid = (int)std::min<uint64_t>((uint64_t)njobs * nchunks, (uint64_t)device_sms() * 8);
    k_cpi_sums<<<grid, COMPACT_THREADS, 0, st>>>(d_jobs, njobs, nchunks);
    k_cpi_scan<<<grid, COMPACT_THREADS, 0, st>>>(d_jobs, njobs, nchunks, d_err);
    k_cpi_totals<<<(njobs + 255) / 256, 256, 0, st>>>(d_jobs, njobs, d_totals);
    return check_launch("k_cpi_count");
}

int launch_cpi_fill(const DevGraph& g, const CpiJob* d_jobs, int njobs, const ScanWork& sw, cudaStream_t st) {
    if (njobs <= 0) return GFD_OK;
    GFD_SCAN_LAUNCH(k_cpi_fill);
    return check_launch("k_cpi_fill");
}

}  // namespace gfd
