// Host-side handles and the engine interface shared by the translation units.
#pragma once

#include <array>
#include <atomic>
#include <mutex>
#include <string>
#include <memory>
#include <vector>

#include "common.cuh"
#include "plan.h"

namespace gfd {
struct Engine;

// The graph's stream-ordered memory pool: destroyed with the last graph or
// result that refers to it (a freed graph gives back what is unused).
struct Pool {
    cudaMemPool_t p = nullptr;
    std::mutex mu;
    cudaStream_t own = nullptr;  // the graph's stream, null once that is gone
    std::vector<void*> dropped;  // memory that a kernel on it may still write
    // Free what was dropped (waits for the graph's stream if there is any).
    void drain() {
        std::lock_guard<std::mutex> lock(mu);
        if (dropped.empty()) return;
        cudaStreamSynchronize(own);
        for (void* q : dropped) cudaFree(q);
        dropped.clear();
    }
    ~Pool() {
        if (p) cudaMemPoolDestroy(p);
        cudaGetLastError();
    }
};

// The end of a call's last kernel, which may still be running when the call returns.
struct Done {
    cudaEvent_t ev = nullptr;
    ~Done() {
        if (ev) cudaEventDestroy(ev);
        cudaGetLastError();
    }
};

// Device memory of the pool shared by results (the short lists of one call) or
// owned by one. Freed without naming a stream, since the call's may be gone by then:
// such a free waits for nothing, and the pool must not hand the memory to another
// stream, or unmap it, under the kernel that writes it. A list that was read is
// written. One dropped unread is waited for by its event, or, written on the graph's
// stream, left to the graph's next call (Pool::drain). An event for every call, and
// the wait for it, took 9 of the 245 us of a small call; frees ordered on the graph's
// stream made small calls back to back 3 times as long.
struct DevBlock {
    void* p = nullptr;
    std::shared_ptr<Pool> pool;
    std::atomic<bool> written{true};
    bool on_own = false;         // by a kernel on the graph's stream
    std::shared_ptr<Done> done;  // else the end of that kernel
    DevBlock(void* q, std::shared_ptr<Pool> from) : p(q), pool(std::move(from)) {}
    DevBlock(void* q, std::shared_ptr<Pool> from, std::shared_ptr<Done> by)
        : p(q), pool(std::move(from)), written(false), on_own(!by), done(std::move(by)) {}
    DevBlock(const DevBlock&) = delete;
    ~DevBlock() {
        if (!written && on_own) {
            std::lock_guard<std::mutex> lock(pool->mu);
            if (pool->own) {
                pool->dropped.push_back(p);
                return;
            }
        }
        if (!written && done && done->ev) cudaEventSynchronize(done->ev);
        cudaFree(p);
        cudaGetLastError();  // a failure here must not surface in a later, unrelated call
    }
};
}

struct gfd_graph {
    int32_t n = 0;
    int64_t m = 0;
    int32_t n_attrs = 0;
    int32_t lbits = 1;
    int64_t bytes = 0;
    gfd::DevGraph dg{};
    std::vector<void*> allocs;
    // per vertex label below the largest one present (others: no vertices)
    std::vector<unsigned long long> label_stats;  // [labels][count, out-degree sum, in-degree sum]
    std::vector<double> moments;                  // [labels][16], see PlanStats
    std::vector<double> moments_all;              // [16]
    std::vector<double> elabel_frac;              // [256]
    // vertices of each label (GFD_WILDCARD: of all) in degree class c: [lo, hi)
    std::vector<std::array<uint32_t, 2 * gfd::N_CLASS>> label_range;
    void range_of(int32_t L, uint32_t* lo, uint32_t* hi) const {
        for (int c = 0; c < gfd::N_CLASS; c++) {
            if (L == GFD_WILDCARD) {
                lo[c] = c ? dg.class_end[c - 1] : 0;
                hi[c] = c < gfd::N_CLASS - 1 ? dg.class_end[c] : (uint32_t)n;
            } else {
                lo[c] = L < n_labels() ? label_range[L][2 * c] : 0;
                hi[c] = L < n_labels() ? label_range[L][2 * c + 1] : 0;
            }
        }
    }
    int32_t n_labels() const { return (int32_t)label_stats.size() / 3; }
    // which: 0 vertices of the label (GFD_WILDCARD: all), 1 their out-degree sum, 2 their in-degree sum
    uint64_t label_stat(int32_t L, int which) const {
        if (L == GFD_WILDCARD) return which == 0 ? (uint64_t)n : (uint64_t)m;
        return L < n_labels() ? label_stats[3 * (size_t)L + which] : 0;
    }
    gfd::PlanStats plan_stats() const {
        gfd::PlanStats p;
        p.n_vertices = n;
        p.n_edges = m;
        p.moments = moments.data();
        p.n_labels = n_labels();
        p.moments_all = moments_all.data();
        p.elabel_frac = elabel_frac.data();
        return p;
    }
    cudaStream_t stream = nullptr;
    gfd::Engine* eng = nullptr;
    std::mutex mu;
    int32_t tuned_variant = -1;          // set by gfd_autotune
    int64_t tuned_budget = 0;
    int32_t tuned_tile_iters = 0;
};

struct gfd_result {
    int32_t k = 0;
    uint64_t n_matches = 0;
    uint64_t n_viol = 0;
    int32_t* d_viol = nullptr;  // device, unsorted, in mem
    std::shared_ptr<gfd::DevBlock> mem;
    int32_t vbits = 32;         // bits of a vertex id
    bool fetched = false;
    std::unique_ptr<int32_t[]> tuples;  // host copy made by gfd_result_tuples
    double prof_ms[5] = {0, 0, 0, 0, 0};
    int64_t prof_launch[5] = {0, 0, 0, 0, 0};
    uint64_t stat[7 + gfd::N_CNT] = {};   // gfd_result_stat: 7 run statistics, then the counters
    cudaStream_t stream = nullptr;
    bool has_cand = false;                      // GFD_FLAG_KEEP_CANDIDATES
    std::vector<std::vector<int32_t>> cand;     // refined candidate list per pattern node
};

namespace gfd {

// ---- job descriptors of the index kernels (device memory)

// The candidates of a bitmap whose adjacency is scanned, shared out as work items
// on the host: the vertices a label has in each degree class are a range [lo, hi)
// (for the wildcard the whole class). An item is an aligned unit of 2^unit(c)
// vertices of class c (ScanLaunch): one hub for a block in class 0, a warp's share
// in the others. A flat range has no adjacency to scan: units of FLAT_UNIT in every
// class, for warps.
struct ScanRange {
    const uint32_t* bm;
    uint32_t lo[N_CLASS], hi[N_CLASS];
    int32_t flat;
};
constexpr int FLAT_UNIT = 10;  // (log2; a lane per word)
__host__ __device__ constexpr uint32_t scan_items(uint32_t lo, uint32_t hi, int unit) {
    return hi <= lo ? 0u : ((hi - 1) >> unit) - (lo >> unit) + 1;
}

struct ScatterJob {      // mark vertices adjacent to the candidates of another level
    ScanRange r;
    const uint32_t* filter;  // only vertices in this bitmap are marked
    uint32_t* marks;
    int32_t scan_out;        // 1: follow out-edges of r, 0: in-edges
    int32_t lab;
};
// out = the vertices of r that are in all marks and, for every constraint, have a
// neighbour (con_dir 1: out-neighbour) in con_bm through an edge with label
// con_lab (or any). out starts as zeros.
struct RefineJob {
    ScanRange r;
    uint32_t* out;
    int32_t nmarks, ncon;
    const uint32_t* marks[2 * MAXK];
    const uint32_t* con_bm[2 * MAXK];
    int8_t con_dir[2 * MAXK];
    int8_t con_any[2 * MAXK];   // con_bm holds vertices of any label
    int16_t con_lab[2 * MAXK];
};
struct CompactJob {      // rank and candidate list of bm
    const uint32_t* bm;
    uint32_t* rank;
    int32_t* cand;           // null: no list wanted
    uint32_t* count;
    uint32_t* csum;          // per-chunk set-bit counts (scratch)
};
struct CpiJob {          // index edges of one spanning-tree edge
    ScanRange r;             // the parent's candidates
    const uint32_t* prank;   // their ranks and number
    const uint32_t* pcount;
    const uint32_t* cbm;
    const uint32_t* crank;
    uint32_t* off;
    int2* idx;               // (position in C(child), vertex id); ids: only the vertex ids (u32)
    int32_t ids;
    uint64_t cap;
    int32_t out;             // 1: children are out-neighbours of the parent candidates
    int32_t lab;
    uint32_t chunk0;         // chunks of the earlier jobs' counts
    uint64_t* csum;          // per-chunk count sums (scratch)
    uint32_t* total;         // number of index edges
};

// One launch of scanning jobs: warp items and block items of all jobs together,
// the units of the classes, and (device memory, apart from the jobs so that a
// search touches few lines) how many items of each kind the earlier jobs have.
struct ScanLaunch {
    uint32_t items = 0, hubs = 0;
    int8_t unit[N_CLASS] = {};
    const uint32_t* first = nullptr;      // [njobs]
    const uint32_t* hub_first = nullptr;  // [njobs]
};
// counting pass: [0] candidates whose adjacency was scanned, [1] adjacency
// entries read (null: not counting)
using ScanCount = unsigned long long*;

// ---- index kernels (index.cu); each launch covers all jobs given
int launch_filter(const DevGraph& g, const FilterKey* d_keys, int nkeys, uint32_t* d_out, cudaStream_t st);
int launch_scatter(const DevGraph& g, const ScatterJob* d_jobs, int njobs, const ScanLaunch& l, ScanCount scan,
                   cudaStream_t st);
int launch_refine(const DevGraph& g, const RefineJob* d_jobs, int njobs, const ScanLaunch& l, ScanCount scan,
                  cudaStream_t st);
// Zeros in the results of the jobs.
int launch_clear(const DevGraph& g, const RefineJob* d_jobs, int njobs, cudaStream_t st);
int launch_compact(const DevGraph& g, const CompactJob* d_jobs, int njobs, cudaStream_t st);
// Index edges in two steps: counts, offsets and per-job totals first, then the
// fill (between the two the caller may read the totals back and allocate exactly).
int launch_cpi_count(const DevGraph& g, const CpiJob* d_jobs, int njobs, const ScanLaunch& l, uint32_t chunks,
                     int32_t* d_err, ScanCount scan, cudaStream_t st);
int launch_cpi_fill(const DevGraph& g, const CpiJob* d_jobs, int njobs, const ScanLaunch& l, ScanCount scan,
                    cudaStream_t st);
uint32_t compact_chunks(const DevGraph& g);
uint32_t cpi_chunks(uint64_t max_parent_candidates);
// units of a launch whose bitmaps have `vertices` vertices in the last class
void scan_units(uint64_t vertices, int most, int8_t* unit);

// ---- enumeration (enumerate.cu)
constexpr int MAX_TILE_ITERS = 64;  // gfd_opts::tile_iters at most: 32 times as many work items per tile
struct EnumArgs {
    DevGraph g;
    const SlotDesc* slots;
    SlotState* state;
    Sched* sched;
    uint32_t* tile_base;  // [3 (n_slots + 1)]: tile prefixes of the fusing, intermediate, last-level slots
    int32_t n_slots;
    int32_t tile;         // largest number of work items per tile
    int32_t n_warps;      // warps of the expansion grid (0: unknown, tiles of `tile`)
    int32_t kmax;         // nodes of the largest pattern a slot may hold
    int32_t narrow;       // steps take no more items than the level to fill has rows
    uint8_t* big;         // N_BIG large frontier buffers of big_bytes each (null: none)
    uint64_t big_bytes;
    uint32_t columns;     // words of a warp's columns in shared memory (set at launch)
};
int enum_init(const EnumArgs& a, cudaStream_t st);
// Mark slots [0, n) idle; start the listed slots (host ids) after their index is built.
int mark_idle(SlotState* state, int n, cudaStream_t st);
int init_slots(const EnumArgs& a, const int* host_ids, int n, cudaStream_t st);
// Capture `steps` enumeration steps (expand + control) into a CUDA graph.
int capture_steps(const EnumArgs& a, int variant, int steps, cudaStream_t st, cudaGraph_t* graph,
                  cudaGraphExec_t* exec);
// Split the violation arena (records [slot, tuple...]) into per-slot lists.
int launch_split(const SlotDesc* slots, const int32_t* arena, uint64_t n, int32_t stride, int32_t* const* lists,
                 unsigned long long* cursor, cudaStream_t st);
// Runs supersteps until every slot is finished. persistent: one cooperative
// launch; else a host loop (optionally captured into CUDA graphs). variant:
// 0 (256 threads, >= 4 blocks/SM), 1 (256, >= 6), 2 (256, >= 8), 3 (128, >= 12),
// 4 (256, >= 5), 5 (512, >= 3).
// general: some slot has a pattern component that starts after level 0 or X
// pushed down (the expansion compiled with those paths); else the leaner one.
// count: the counting instantiation (persistent, general, 256 threads), which
// also fills Sched::cnt; used untimed for the algorithmic-byte model.
int enum_run(const EnumArgs& a, bool persistent, bool use_graph, int variant, bool general, cudaStream_t st,
             cudaEvent_t ev0, cudaEvent_t ev1, int64_t* launches, bool count = false);
int variant_threads(int variant);
constexpr int N_VARIANTS = 6;

// ---- orchestration (run.cu)
// SM count of the current device (queried once per device; 1 if the query
// fails, and the next launch then reports the error).
int device_sms();

int graph_load(const gfd_graph_desc* d, const gfd_opts* o, gfd_graph** out);
void graph_free(gfd_graph* g);
void engine_free(Engine* e);
// narrow: no step takes more items than the level that it fills has rows, and no
// large buffers (the second run of a call in which such a step did not come out).
int run_batch(gfd_graph* g, const gfd_gfd* const* phis, int32_t n, const gfd_opts* o, gfd_result** out,
              bool narrow = false);
int session_create(gfd_graph* g, int32_t max_slots, const gfd_opts* o, gfd_session** out);
void session_free(gfd_session* s);
int session_submit(gfd_session* s, const gfd_gfd* phi, int64_t* id);
int session_step(gfd_session* s, int32_t* n_advanced, int32_t* n_running, int32_t* n_queued);
int session_next_result(gfd_session* s, int64_t* id, gfd_result** out);
int session_cancel(gfd_session* s, int64_t id);
double session_stat(const gfd_session* s, int32_t which);
int autotune(gfd_graph* g, const gfd_gfd* const* phis, int32_t n, const gfd_opts* o, gfd_opts* best);
// Sort the violation tuples on the device and copy them to dst (host memory,
// n_viol * k ints); result_fetch does this into the result's own buffer.
int result_sort_copy(gfd_result* r, int32_t* dst);
// The same for n results at once, into one host buffer: result 0's tuples,
// then result 1's, ... (one device sort keyed by (result, tuple), one copy).
int results_sort_copy(gfd_result* const* rs, int n, int32_t* out, uint64_t capacity);
int result_fetch(gfd_result* r);

}  // namespace gfd
