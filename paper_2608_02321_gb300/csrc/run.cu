// Orchestration of validation runs: batches (gfd_validate, gfd_validate_batch)
// and continuous-batching serving sessions (gfd_session_*).
//
// Device memory is organised in two kinds of blocks:
//   - slot tables (one per run or session): a SlotDesc and a SlotState per GFD
//     slot, the scheduler state, the per-step tile prefix and, for batch runs,
//     the shared violation arena;
//   - one workspace per group of GFDs admitted together: candidate bitmaps,
//     ranks and lists, index edges, partial-match buffers, index-build job
//     tables and scratch.
// For a group the host plans every GFD (plan.cpp), deduplicates candidate-filter
// keys across the group (the shared candidate cache), derives every buffer's
// capacity from the graph's per-label statistics, allocates the workspace from
// the graph's stream-ordered pool, uploads descriptors and job tables, and
// launches one filter pass for all keys plus the refinement and index phases
// (each launch covers every GFD of the group). Nothing waits on the host until
// the counters are read back at the end.
#include <cub/cub.cuh>

#include <algorithm>
#include <array>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <memory>
#include <unordered_map>
#include <vector>

#include "engine.h"

namespace gfd {

struct Engine {
    std::shared_ptr<Pool> pool;
};

void engine_free(Engine* e) {
    if (!e) return;
    if (e->pool) {
        // results may keep the pool itself; what they free from now on is written
        std::lock_guard<std::mutex> lock(e->pool->mu);
        if (e->pool->own) cudaStreamSynchronize(e->pool->own);
        e->pool->own = nullptr;
        for (void* q : e->pool->dropped) cudaFree(q);
        e->pool->dropped.clear();
        cudaMemPoolTrimTo(e->pool->p, 0);
    }
    cudaGetLastError();
    delete e;
}

namespace {

constexpr int PROF_FILTER = 0, PROF_REFINE = 1, PROF_INDEX = 2, PROF_ENUM = 3;

struct Layout {
    size_t size = 256;  // offset 0 is reserved
    size_t take(size_t bytes) {
        size_t off = size;
        size = (size + bytes + 255) & ~(size_t)255;
        return off;
    }
};

int get_pool(gfd_graph* g, std::shared_ptr<Pool>* out) {
    if (!g->eng) g->eng = new Engine();
    if (!g->eng->pool) {
        int dev = 0;
        GFD_CUDA(cudaGetDevice(&dev));
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        auto pool = std::make_shared<Pool>();
        GFD_CUDA(cudaMemPoolCreate(&pool->p, &props));
        uint64_t thr = UINT64_MAX;
        GFD_CUDA(cudaMemPoolSetAttribute(pool->p, cudaMemPoolAttrReleaseThreshold, &thr));
        pool->own = g->stream;
        g->eng->pool = std::move(pool);
    }
    *out = g->eng->pool;
    return GFD_OK;
}

int pool_alloc(cudaMemPool_t pool, size_t bytes, cudaStream_t st, void** out, const char* what) {
    cudaError_t e = cudaMallocFromPoolAsync(out, std::max<size_t>(bytes, 256), pool, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *out = nullptr;
        set_error(GFD_ERR_OUT_OF_MEMORY, "%s: %zu device bytes: %s", what, bytes, cudaGetErrorString(e));
        return GFD_ERR_OUT_OF_MEMORY;
    }
    return GFD_OK;
}

uint64_t env_u64(const char* name, uint64_t dflt) {
    const char* s = getenv(name);
    if (!s || !*s) return dflt;
    return strtoull(s, nullptr, 10);
}

struct ProfEvents {
    bool on = false;
    cudaEvent_t ev[2 * 5] = {};
    ~ProfEvents() {
        for (auto e : ev)
            if (e) cudaEventDestroy(e);
    }
    int init(bool enable) {
        on = enable;
        if (!on) return GFD_OK;
        for (auto& e : ev) GFD_CUDA(cudaEventCreate(&e));
        return GFD_OK;
    }
    void begin(int w, cudaStream_t st) {
        if (on) cudaEventRecord(ev[2 * w], st);
    }
    void end(int w, cudaStream_t st) {
        if (on) cudaEventRecord(ev[2 * w + 1], st);
    }
    double ms(int w) {
        if (!on) return 0;
        float t = 0;
        if (cudaEventElapsedTime(&t, ev[2 * w], ev[2 * w + 1]) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return t;
    }
};

}  // namespace

// ------------------------------------------------------------------ slot tables
struct Tables {
    int max_slots = 0;
    uint8_t* base = nullptr;
    SlotDesc* desc = nullptr;
    SlotState* state = nullptr;
    Sched* sched = nullptr;
    uint32_t* tiles = nullptr;
    int32_t* err = nullptr;
    int32_t** vptr = nullptr;
    unsigned long long* vcur = nullptr;
    int32_t* varena = nullptr;  // batch runs only
    uint64_t vcap = 0;
    int vstride = 0;
    int32_t tile = 2048;
};

namespace {

int tables_alloc(cudaMemPool_t pool, int max_slots, int block_threads, int tile_iters, int kmax_arena,
                 uint64_t vcap, bool bounded_run, cudaStream_t st, Tables* T) {
    Layout L;
    const size_t o_desc = L.take(sizeof(SlotDesc) * max_slots);
    const size_t o_state = L.take(sizeof(SlotState) * max_slots);
    const size_t o_sched = L.take(sizeof(Sched));
    const size_t o_tiles = L.take(4ull * 3 * (max_slots + 1));  // three tile prefixes
    const size_t o_err = L.take(4);
    const size_t zero_end = L.size;
    const size_t o_vptr = L.take(sizeof(int32_t*) * max_slots);
    const size_t o_vcur = L.take(8ull * max_slots);
    const int vstride = kmax_arena + 1;
    const size_t o_arena = kmax_arena > 0 ? L.take(4ull * vstride * vcap) : 0;
    void* base = nullptr;
    if (int rc = pool_alloc(pool, L.size, st, &base, "slot tables")) return rc;
    T->max_slots = max_slots;
    T->base = (uint8_t*)base;
    T->desc = (SlotDesc*)(T->base + o_desc);
    T->state = (SlotState*)(T->base + o_state);
    T->sched = (Sched*)(T->base + o_sched);
    T->tiles = (uint32_t*)(T->base + o_tiles);
    T->err = (int32_t*)(T->base + o_err);
    T->vptr = (int32_t**)(T->base + o_vptr);
    T->vcur = (unsigned long long*)(T->base + o_vcur);
    T->varena = kmax_arena > 0 ? (int32_t*)(T->base + o_arena) : nullptr;
    T->vcap = kmax_arena > 0 ? vcap : 0;
    T->vstride = vstride;
    T->tile = 32 * tile_iters;  // work items per warp visit
    GFD_CUDA(cudaMemsetAsync(T->base + o_desc, 0, zero_end - o_desc, st));
    Sched s{};
    s.n_slots = max_slots;
    s.tile = (uint32_t)T->tile;
    s.timeout_ns = env_u64("GFD_WAIT_LIMIT_MS", 10000) * 1000000ull;
    // a run as a whole is bounded in time; a session's host drives bounded
    // rounds of steps and has no overall limit
    s.run_limit_ns = bounded_run ? env_u64("GFD_RUN_LIMIT_MS", 600000) * 1000000ull : UINT64_MAX;
    s.varena = T->varena;
    s.varena_cap = T->vcap;
    s.vstride = vstride;
    GFD_CUDA(cudaMemcpyAsync(T->sched, &s, sizeof(s), cudaMemcpyHostToDevice, st));
    return GFD_OK;
}

EnumArgs enum_args(const gfd_graph* g, const Tables& T, int kmax) {
    EnumArgs A;
    A.g = g->dg;
    A.slots = T.desc;
    A.state = T.state;
    A.sched = T.sched;
    A.tile_base = T.tiles;
    A.n_slots = T.max_slots;
    A.tile = T.tile;
    A.n_warps = 0;
    A.kmax = kmax;
    A.narrow = 0;
    A.big = nullptr;
    A.big_bytes = 0;
    A.columns = 0;
    return A;
}

// ------------------------------------------------------------------ groups
struct Phase {
    int kind;  // 0 scatter, 1 refine, 2 clear results, 3 clear marks
    size_t first, count;
    ScanLaunch launch;
};

// The refinement of a group, planned before any pointer is known. Bitmaps are
// written once and known by number: [0, keys) the candidate filters', then the
// refinements' results. A result is determined by its source, its constraints and
// the bitmaps they look at, so GFDs of the group that refine the same candidates
// in the same way (and nodes of one GFD that look alike) share it, and everything
// built from it: rank, candidate list and index edges.
struct ConSpec {
    int bm;       // neighbours wanted in this bitmap
    int dir;      // 1: out-neighbours
    int lab;
    bool gather;  // looked up from the candidates; else marked from bm's vertices
};
struct RefineSpec {
    int src, dst;
    std::vector<ConSpec> cons;
};
struct IndexSpec {
    int parent, child;  // final bitmaps (Group::finals)
    int dir, lab;
    bool ids;           // for a last level: vertex ids alone
    uint64_t bound;     // most index edges there can be
    size_t entry() const { return ids ? 4 : 8; }
};
struct VecHash {
    size_t operator()(const std::vector<int32_t>& v) const {
        uint64_t h = 1469598103934665603ull;
        for (int32_t x : v) h = (h ^ (uint32_t)x) * 1099511628211ull;
        return (size_t)(h ^ (h >> 32));
    }
};
using VecMap = std::unordered_map<std::vector<int32_t>, int, VecHash>;

}  // namespace

struct Group {
    int n = 0;
    std::vector<int> slot;
    std::vector<HostPlan> plans;
    std::vector<SlotDesc> descs;
    std::vector<FilterKey> keys;
    std::vector<int> bm_key;                 // the filter key (so the label) of each bitmap
    std::vector<RefineSpec> refines;         // in launch order
    std::vector<size_t> phase_end;           // refines of each phase end here
    size_t n_marks = 0;
    bool reuse = false;                      // bitmaps and marks take the place of ones no longer read
    std::vector<int> place;                  // of each refinement's result
    size_t n_places = 0, n_mark_places = 0;
    std::vector<int> finals;                 // bitmaps that are some level's candidates
    std::vector<char> final_list;            // a candidate list is wanted
    std::vector<std::array<int, MAXK>> level_final, level_index;  // per (GFD, level)
    std::vector<IndexSpec> index;
    uint8_t* base = nullptr;
    size_t bytes = 0;
    struct Off {
        size_t rows[MAXK], wpre[MAXK];
    };
    std::vector<Off> offs;
    std::vector<size_t> o_rank, o_cand;      // per final
    std::vector<size_t> o_off, o_idx;        // per index (o_idx only when in the workspace)
    size_t o_keybm = 0, o_zero = 0, o_zero_end = 0, o_counts = 0, o_bm = 0, o_marks = 0;
    size_t o_cmp_sums = 0, o_cpi_sums = 0, o_cpi_tot = 0;
    uint64_t big_bytes = 0;       // each large frontier buffer (0: none)
    size_t o_big = 0;
    bool idx_inside = false;      // index edges in the workspace, at their bound
    uint8_t* cpi_base = nullptr;  // else: allocated exactly after counting
    size_t cpi_bytes = 0;
    size_t cpi_bound = 0;  // upper bound of cpi_bytes known at planning time
    size_t o_jobs = 0, o_keys = 0, o_first = 0, o_cmp = 0, o_sct = 0, o_ref = 0, o_cpi = 0, jobs_end = 0;
    uint32_t cmp_chunks = 1, cpi_nch = 0;
    std::vector<CompactJob> compact_jobs;
    std::vector<ScatterJob> scatter_jobs;
    std::vector<RefineJob> refine_jobs;
    std::vector<CpiJob> cpi_jobs;
    std::vector<uint32_t> first;  // ScanLaunch::first and hub_first of all launches
    std::vector<Phase> phases;
    ScanLaunch cpi_launch;
    std::vector<SlotState> state_img;  // host image of the cleared states (kept until copied)
    int live = 0;  // slots of this group still running (sessions)
};

namespace {

// Index edges up to this many bytes (their bound, from degree sums) are part of
// the workspace: no read-back of the counts, no second allocation. Beyond, the
// counts are read back (one synchronisation) and exactly as much is allocated.
constexpr size_t IDX_INSIDE = (size_t)1 << 30;
// A session's requests hold their memory while they run and share a budget, so there
// the bound may be a sixteenth of the rest of the workspace at most: with more, fewer
// requests ran at once (their index edges are often a small part of the bound). A call
// whose workspace cannot be had is planned again without such room.
constexpr size_t SESSION_IDX_SHARE = 16;
enum class Room { AMPLE, SESSION, LEAN };

// Refinement results and marks up to this many bytes lie apart and are cleared by one
// call. Beyond, a phase's results take the places of bitmaps that no later phase reads,
// its marks those of the phase before, and each phase clears its own (the same bytes
// in all, but two more launches a phase: 32 GFDs on 5M vertices, 190 MB, 6.34 -> 6.43
// ms): the workspace of 256 GFDs over labels of 0.1 and
// 4 % of 16M vertices, without partial matches, has 14.1 instead of 18.1 GB.
constexpr size_t BITMAPS_APART = (size_t)256 << 20;

// Largest units (log2 of vertices) of the adjacency scans, see scan_units.
constexpr int REFINE_UNIT = 8;
constexpr int INDEX_UNIT = 10;

// Violation lists up to this many bytes share one allocation per call (which
// lives until the last of their results is freed); larger ones have their own.
constexpr size_t SHARED_LIST = 64 << 10;

// Top-down constraint "x in C(i) needs a neighbour in C(q) through an edge
// leaving x (dir 1) or entering x (dir 0)": scattering from C(q) scans the
// opposite-direction adjacency of the q label class; gathering scans the
// dir-direction adjacency of the i label class but stops at the first hit
// (counted as half of it).
bool td_gather_cheaper(const gfd_graph* g, int32_t label_q, int32_t label_i, int dir) {
    auto degsum = [&](int32_t L, bool out) { return (double)g->label_stat(L, out ? 1 : 2); };
    const double scatter = degsum(label_q, dir == 0);
    const double gather = 0.5 * degsum(label_i, dir == 1);
    return gather < scatter;
}

// Plans, capacities and the workspace layout of a group (host only). With
// strict_budget, a frontier_per_slot that cannot hold MIN_CHUNK partial matches
// at every level of some GFD is an error instead of being raised to that.
constexpr uint64_t BIG_MIN_CHUNK = 1 << 16;
constexpr uint64_t MIN_CHUNK = 1024;
// rows are counted in 24 bits; warps that find no room may still add theirs (at
// most 32 each)
constexpr uint64_t MAX_CHUNK = (1ull << 24) - (1ull << 20);
int group_plan(gfd_graph* g, const gfd_gfd* const* phis, int n, const gfd_opts* o, int64_t frontier_per_slot,
               Group* G, bool strict_budget = false, bool with_big = false, Room room = Room::AMPLE) {
    const uint32_t nwords = g->dg.nwords;
    G->n = n;
    G->plans.resize(n);
    for (int s = 0; s < n; s++)
        if (int rc = make_plan(phis[s], g->n_attrs, g->plan_stats(), &G->plans[s],
                               !(o && (o->flags & GFD_FLAG_NON_INDUCED)), o && (o->flags & GFD_FLAG_PUSH_X)))
            return rc;
    VecMap key_id;
    std::vector<std::array<int, MAXK>> cur(n);  // per (GFD, level): the bitmap that holds its candidates so far
    for (int s = 0; s < n; s++)
        for (int i = 0; i < G->plans[s].k; i++) {
            const FilterKey& K = G->plans[s].key[i];
            std::vector<int32_t> t = {K.label, (int32_t)K.dout_min, (int32_t)K.din_min, K.self_exp, K.n_attr};
            for (int a = 0; a < K.n_attr; a++) {
                t.push_back(K.attr_a[a]);
                t.push_back(K.attr_c[a]);
            }
            const auto it = key_id.emplace(std::move(t), (int)G->keys.size());
            if (it.second) {
                G->bm_key.push_back((int)G->keys.size());
                G->keys.push_back(K);
            }
            cur[s][i] = it.first->second;
        }
    const int nkeys = (int)G->keys.size();
    auto lab_count = [&](int32_t L) { return g->label_stat(L, 0); };
    auto lab_deg = [&](int32_t L, bool outdir) { return g->label_stat(L, outdir ? 1 : 2); };
    // refinement: top-down level by level, then bottom-up. Each constraint is
    // applied in the cheaper direction: marks from the other level's candidates
    // (cost ~ their degree sum), or a look from the level's own candidates that
    // stops at the first hit.
    VecMap done;
    auto refine_level = [&](int s, int lvl, const std::vector<Con>& cons) {
        if (cons.empty()) return;
        const HostPlan& P = G->plans[s];
        RefineSpec R;
        R.src = cur[s][lvl];
        std::vector<int32_t> t = {R.src};
        for (const Con& c : cons) {
            const bool gather = td_gather_cheaper(g, P.key[c.q].label, P.key[lvl].label, c.dir);
            R.cons.push_back({cur[s][c.q], c.dir, c.lab, gather});
            t.insert(t.end(), {cur[s][c.q], c.dir, c.lab, gather});
        }
        const auto it = done.emplace(std::move(t), (int)G->bm_key.size());
        if (it.second) {
            R.dst = (int)G->bm_key.size();
            G->bm_key.push_back(G->bm_key[R.src]);
            for (const ConSpec& c : R.cons) G->n_marks += !c.gather;
            G->refines.push_back(std::move(R));
        }
        cur[s][lvl] = it.first->second;
    };
    int maxk = 0;
    for (auto& P : G->plans) maxk = std::max(maxk, P.k);
    auto end_phase = [&] {
        if (G->refines.size() > (G->phase_end.empty() ? 0 : G->phase_end.back())) G->phase_end.push_back(G->refines.size());
    };
    if (!(o && (o->flags & GFD_FLAG_NO_REFINE))) {
        for (int lvl = 0; lvl < maxk; lvl++) {
            for (int s = 0; s < n; s++)
                if (lvl < G->plans[s].k) refine_level(s, lvl, G->plans[s].td[lvl]);
            end_phase();
        }
        for (int lvl = maxk - 1; lvl >= 0; lvl--) {
            for (int s = 0; s < n; s++)
                if (lvl < G->plans[s].k) refine_level(s, lvl, G->plans[s].bu[lvl]);
            end_phase();
        }
    }
    // the levels' final bitmaps, and the index edges of the spanning trees
    std::vector<int> final_of(G->bm_key.size(), -1);
    G->level_final.resize(n);
    G->level_index.resize(n);
    VecMap index_id;
    for (int s = 0; s < n; s++) {
        const HostPlan& P = G->plans[s];
        for (int i = 0; i < P.k; i++) {
            int& f = final_of[cur[s][i]];
            if (f < 0) {
                f = (int)G->finals.size();
                G->finals.push_back(cur[s][i]);
                G->final_list.push_back(0);
            }
            G->level_final[s][i] = f;
            // lists are read for roots, levels that start a component, and by request
            if (i == 0 || P.lv[i].par < 0 || (o && (o->flags & GFD_FLAG_KEEP_CANDIDATES))) G->final_list[f] = 1;
        }
        for (int i = 1; i < P.k; i++) {
            const int par = P.lv[i].par;
            if (par < 0) continue;  // starts a component: no index edges
            const int pf = G->level_final[s][par], cf = G->level_final[s][i];
            const auto it = index_id.emplace(std::vector<int32_t>{pf, cf, P.lv[i].tdir, P.lv[i].tlab, i == P.k - 1},
                                             (int)G->index.size());
            if (it.second) {
                const int32_t plab = P.key[par].label;
                G->index.push_back({pf, cf, P.lv[i].tdir, P.lv[i].tlab, i == P.k - 1,
                                    std::min<uint64_t>(lab_deg(plab, P.lv[i].tdir == 1), (uint64_t)g->m)});
            }
            G->level_index[s][i] = it.first->second;
        }
    }
    // where the refinements' results and marks lie
    const size_t bm_bytes = 4ull * nwords, n_results = G->refines.size();
    G->reuse = bm_bytes * (n_results + G->n_marks) > (room == Room::LEAN ? 0 : BITMAPS_APART);
    G->place.resize(n_results);
    if (!G->reuse) {
        for (size_t i = 0; i < n_results; i++) G->place[i] = (int)i;
        G->n_places = n_results;
        G->n_mark_places = G->n_marks;
    } else {
        const size_t phases = G->phase_end.size();
        std::vector<size_t> last(G->bm_key.size(), 0);  // the last phase that reads (or writes) each bitmap
        for (size_t p = 0, i = 0; p < phases; p++)
            for (; i < G->phase_end[p]; i++) {
                const RefineSpec& R = G->refines[i];
                last[R.src] = last[R.dst] = p;
                for (const ConSpec& c : R.cons) last[c.bm] = p;
            }
        for (int f : G->finals) last[f] = phases;
        std::vector<std::vector<int>> over(phases + 1);  // places that are free after each phase
        std::vector<int> free_places;
        for (size_t p = 0, i = 0; p < phases; p++) {
            if (p) free_places.insert(free_places.end(), over[p - 1].begin(), over[p - 1].end());
            size_t marks = 0;
            for (; i < G->phase_end[p]; i++) {
                if (free_places.empty()) {
                    G->place[i] = (int)G->n_places++;
                } else {
                    G->place[i] = free_places.back();
                    free_places.pop_back();
                }
                over[last[G->refines[i].dst]].push_back(G->place[i]);
                for (const ConSpec& c : G->refines[i].cons) marks += !c.gather;
            }
            G->n_mark_places = std::max(G->n_mark_places, marks);
        }
    }
    Layout L;
    G->descs.assign(n, SlotDesc{});
    G->offs.resize(n);
    // A quarter of a batch's frontier budget goes to the N_BIG large buffers when
    // the GFDs are many and their own shares stay large without it. Batch of 256
    // GFDs on 4M vertices with 48 GiB: 443 steps -> 49, enumeration 172 -> 147 ms
    // (its last slots, with 1/256 of the budget each, took 435 of the steps). Below 13
    // GFDs a large buffer, 1/16 of the budget, is no larger than their own shares of
    // the other three quarters (and would have to exceed the budget to be).
    size_t big_need = 0;
    uint64_t widest = 0;
    for (auto& P : G->plans) {
        uint64_t b = 0;
        for (int l = 1; l <= P.k - 2; l++) b += 4ull * row_width(l) + 8;
        widest = std::max(widest, b);
    }
    const bool big = with_big && n > 3 * N_BIG && !(o && o->chunk_rows > 0) && widest &&
                     (uint64_t)frontier_per_slot / 4 * 3 / widest >= BIG_MIN_CHUNK;
    if (big) {
        G->big_bytes = (uint64_t)frontier_per_slot * n / (4 * N_BIG) & ~(uint64_t)255;
        frontier_per_slot = frontier_per_slot / 4 * 3;
    }
    for (int s = 0; s < n; s++) {
        const HostPlan& P = G->plans[s];
        SlotDesc& D = G->descs[s];
        memset(&D, 0, sizeof(D));
        D.k = P.k;
        D.nx = P.nx;
        D.ny = P.ny;
        D.y_false = P.y_false;
        D.push_x = P.push_x ? 1 : 0;
        for (int i = 0; i < P.k; i++) {
            D.order[i] = P.order[i];
            D.lv[i] = P.lv[i];
        }
        for (size_t q = 0; q < P.lits.size(); q++) D.lit[q] = P.lits[q];
        uint64_t row_bytes = 0;
        for (int l = 1; l <= P.k - 2; l++) row_bytes += 4ull * row_width(l) + 8;
        uint64_t chunk = o && o->chunk_rows > 0 ? (uint64_t)o->chunk_rows
                                                : (row_bytes ? (uint64_t)frontier_per_slot / row_bytes : MAX_CHUNK);
        if (strict_budget && !(o && o->chunk_rows > 0) && chunk < MIN_CHUNK) {
            set_error(GFD_ERR_OUT_OF_MEMORY,
                      "frontier budget of %lld bytes per GFD holds fewer than %llu partial matches per level of GFD "
                      "%d (it needs %llu bytes)",
                      (long long)frontier_per_slot, (unsigned long long)MIN_CHUNK, s,
                      (unsigned long long)(MIN_CHUNK * row_bytes));
            return GFD_ERR_OUT_OF_MEMORY;
        }
        chunk = std::max<uint64_t>(MIN_CHUNK, std::min<uint64_t>(chunk, MAX_CHUNK));
        D.chunk = chunk;
        Group::Off& F = G->offs[s];
        if (big && row_bytes) {
            Layout B;
            B.size = 0;
            D.big_chunk = std::max(chunk, std::min<uint64_t>(MAX_CHUNK, (G->big_bytes - 256 * 2 * MAXK) / row_bytes));
            for (int l = 1; l <= P.k - 2; l++) {
                D.big_rows[l] = B.take(4ull * row_width(l) * D.big_chunk);
                D.big_wpre[l] = B.take(8ull * D.big_chunk);
            }
            big_need = std::max(big_need, B.size);
        }
        for (int l = 1; l <= P.k - 2; l++) {
            F.rows[l] = L.take(4ull * row_width(l) * chunk);
            F.wpre[l] = L.take(8ull * chunk);
        }
    }
    if (big) {
        G->big_bytes = big_need;
        G->o_big = L.take(G->big_bytes * N_BIG);
    }
    auto label_of = [&](int bm) { return G->keys[G->bm_key[bm]].label; };
    G->o_keybm = L.take(bm_bytes * std::max(1, nkeys));
    // zeroed by one call: the finals' counts, the refinements' results and marks
    // (results and marks by each phase when they take turns)
    G->o_zero = L.size;
    G->o_counts = L.take(4ull * G->finals.size());
    if (G->reuse) G->o_zero_end = L.size;
    G->o_bm = L.take(bm_bytes * G->n_places);
    G->o_marks = L.take(bm_bytes * G->n_mark_places);
    if (!G->reuse) G->o_zero_end = L.size;
    for (size_t f = 0; f < G->finals.size(); f++) {
        G->o_rank.push_back(L.take(bm_bytes));
        G->o_cand.push_back(G->final_list[f] ? L.take(4ull * std::max<uint64_t>(1, lab_count(label_of(G->finals[f])))) : 0);
    }
    for (const IndexSpec& X : G->index) {
        const uint64_t cap = lab_count(label_of(G->finals[X.parent]));
        G->o_off.push_back(L.take(4ull * (cap + 1)));
        G->cpi_nch += cpi_chunks(cap);
        G->cpi_bound += X.entry() * std::max<uint64_t>(1, X.bound) + 256;
    }
    G->cmp_chunks = compact_chunks(g->dg);
    G->o_cmp_sums = L.take(4ull * G->cmp_chunks * G->finals.size());
    G->o_cpi_sums = L.take(8ull * std::max<uint32_t>(1, G->cpi_nch));
    G->o_cpi_tot = L.take(4ull * std::max<size_t>(1, G->index.size()));
    G->idx_inside = room != Room::LEAN &&
                    G->cpi_bound <= (room == Room::SESSION ? std::min(IDX_INSIDE, L.size / SESSION_IDX_SHARE) : IDX_INSIDE);
    if (G->idx_inside)
        for (const IndexSpec& X : G->index) G->o_idx.push_back(L.take(X.entry() * std::max<uint64_t>(1, X.bound)));
    // the region uploaded from the host: keys and job tables
    G->o_jobs = L.size;
    G->o_keys = L.take(sizeof(FilterKey) * std::max(1, nkeys));
    G->o_cmp = L.take(sizeof(CompactJob) * std::max<size_t>(1, G->finals.size()));
    G->o_sct = L.take(sizeof(ScatterJob) * std::max<size_t>(1, G->n_marks));
    G->o_ref = L.take(sizeof(RefineJob) * std::max<size_t>(1, G->refines.size()));
    G->o_cpi = L.take(sizeof(CpiJob) * std::max<size_t>(1, G->index.size()));
    G->o_first = L.take(8ull * (G->n_marks + G->refines.size() + G->index.size()));
    G->jobs_end = L.size;
    G->bytes = L.size;
    return GFD_OK;
}

// Absolute pointers, job tables and their upload; the descriptors go to the
// slot tables at the group's slots, whose states are cleared.
int group_build(gfd_graph* g, Group* G, const Tables& T, cudaStream_t st) {
    const size_t bm_bytes = 4ull * g->dg.nwords;
    const int nkeys = (int)G->keys.size();
    uint8_t* base = G->base;
    const int n = G->n;
    auto bitmap = [&](int id) {
        return (uint32_t*)(base + (id < nkeys ? G->o_keybm + bm_bytes * id : G->o_bm + bm_bytes * G->place[id - nkeys]));
    };
    auto label_of = [&](int bm) { return G->keys[G->bm_key[bm]].label; };
    // a job's share of a launch: its items come after those of the jobs before it
    auto range_of = [&](int bm, bool flat) {
        ScanRange r{};
        r.bm = bitmap(bm);
        r.flat = flat;
        g->range_of(label_of(bm), r.lo, r.hi);
        return r;
    };
    // (64-bit sums: a launch of more than 2^32 items is refused)
    auto lay_out = [&](auto* jobs, size_t count, int most, ScanLaunch* l) -> int {
        uint64_t vertices = 0, items = 0, hubs = 0;
        for (size_t j = 0; j < count; j++)
            if (!jobs[j].r.flat) vertices += jobs[j].r.hi[N_CLASS - 1] - jobs[j].r.lo[N_CLASS - 1];
        scan_units(vertices, most, l->unit);
        const size_t at = G->first.size();
        G->first.resize(at + 2 * count);
        l->first = (const uint32_t*)(base + G->o_first) + at;
        l->hub_first = l->first + count;
        for (size_t j = 0; j < count; j++) {
            const ScanRange& r = jobs[j].r;
            G->first[at + j] = (uint32_t)items;
            G->first[at + count + j] = (uint32_t)hubs;
            for (int c = 0; c < N_CLASS; c++) {
                const uint32_t k = scan_items(r.lo[c], r.hi[c], r.flat ? FLAT_UNIT : l->unit[c]);
                if (c == 0 && !r.flat) hubs += k;
                else items += k;
            }
        }
        if (items > 0xffffffffull || hubs > 0xffffffffull) {
            set_error(GFD_ERR_UNSUPPORTED, "index build of %d GFDs has more than 2^32 work items (split the batch)", n);
            return GFD_ERR_UNSUPPORTED;
        }
        l->items = (uint32_t)items;
        l->hubs = (uint32_t)hubs;
        return GFD_OK;
    };
    size_t from = 0;
    uint32_t* next_marks = (uint32_t*)(base + G->o_marks);
    for (size_t end : G->phase_end) {
        Phase sc{0, G->scatter_jobs.size(), 0, {}}, rf{1, G->refine_jobs.size(), 0, {}};
        if (G->reuse) next_marks = (uint32_t*)(base + G->o_marks);
        for (size_t i = from; i < end; i++) {
            const RefineSpec& R = G->refines[i];
            RefineJob J{};
            J.out = bitmap(R.dst);
            for (const ConSpec& c : R.cons) {
                if (c.gather) {
                    J.con_bm[J.ncon] = bitmap(c.bm);
                    J.con_dir[J.ncon] = (int8_t)c.dir;
                    J.con_lab[J.ncon] = (int16_t)c.lab;
                    J.con_any[J.ncon] = label_of(c.bm) == GFD_WILDCARD;
                    J.ncon++;
                    continue;
                }
                ScatterJob S{};
                S.r = range_of(c.bm, false);
                S.filter = bitmap(R.src);
                S.marks = next_marks;
                // x needs an out-neighbour y in C(q) (x -> y): follow in-edges of y
                S.scan_out = c.dir ? 0 : 1;
                S.lab = c.lab;
                G->scatter_jobs.push_back(S);
                J.marks[J.nmarks++] = next_marks;
                next_marks += g->dg.nwords;
            }
            J.r = range_of(R.src, J.ncon == 0);
            G->refine_jobs.push_back(J);
        }
        from = end;
        sc.count = G->scatter_jobs.size() - sc.first;
        rf.count = G->refine_jobs.size() - rf.first;
        if (int rc = lay_out(G->scatter_jobs.data() + sc.first, sc.count, REFINE_UNIT, &sc.launch)) return rc;
        if (int rc = lay_out(G->refine_jobs.data() + rf.first, rf.count, REFINE_UNIT, &rf.launch)) return rc;
        if (G->reuse) {
            G->phases.push_back({2, rf.first, rf.count, {}});
            if (sc.count) G->phases.push_back({3, 0, sc.count, {}});
        }
        if (sc.count) G->phases.push_back(sc);
        G->phases.push_back(rf);
    }
    auto rank_of = [&](int f) { return (uint32_t*)(base + G->o_rank[f]); };
    auto count_of = [&](int f) { return (uint32_t*)(base + G->o_counts) + f; };
    for (size_t f = 0; f < G->finals.size(); f++) {
        CompactJob J{};
        J.bm = bitmap(G->finals[f]);
        J.rank = rank_of((int)f);
        J.cand = G->final_list[f] ? (int32_t*)(base + G->o_cand[f]) : nullptr;
        J.count = count_of((int)f);
        J.csum = (uint32_t*)(base + G->o_cmp_sums + 4ull * G->cmp_chunks * f);
        G->compact_jobs.push_back(J);
    }
    uint32_t chunk = 0;
    for (size_t x = 0; x < G->index.size(); x++) {
        const IndexSpec& X = G->index[x];
        CpiJob J{};
        J.r = range_of(G->finals[X.parent], false);
        J.prank = rank_of(X.parent);
        J.pcount = count_of(X.parent);
        J.cbm = bitmap(G->finals[X.child]);
        J.crank = rank_of(X.child);
        J.off = (uint32_t*)(base + G->o_off[x]);
        J.idx = G->idx_inside ? (int2*)(base + G->o_idx[x]) : nullptr;
        J.ids = X.ids;
        J.cap = X.bound;
        J.out = X.dir;
        J.lab = X.lab;
        J.chunk0 = chunk;
        J.csum = (uint64_t*)(base + G->o_cpi_sums) + chunk;
        J.total = (uint32_t*)(base + G->o_cpi_tot) + x;
        chunk += cpi_chunks(g->label_stat(label_of(G->finals[X.parent]), 0));
        G->cpi_jobs.push_back(J);
    }
    if (int rc = lay_out(G->cpi_jobs.data(), G->cpi_jobs.size(), INDEX_UNIT, &G->cpi_launch)) return rc;
    for (int s = 0; s < n; s++) {
        const HostPlan& P = G->plans[s];
        SlotDesc& D = G->descs[s];
        const Group::Off& F = G->offs[s];
        for (int i = 0; i < P.k; i++) {
            const int f = G->level_final[s][i];
            D.bm[i] = bitmap(G->finals[f]);
            D.rank[i] = rank_of(f);
            D.cand[i] = G->final_list[f] ? (int32_t*)(base + G->o_cand[f]) : nullptr;
            D.cand_n[i] = count_of(f);
            if (i >= 1 && P.lv[i].par >= 0) {
                D.cpi_off[i] = G->cpi_jobs[G->level_index[s][i]].off;
                D.cpi_idx[i] = G->cpi_jobs[G->level_index[s][i]].idx;  // null until the index edges are counted
            }
        }
        for (int l = 1; l <= P.k - 2; l++) {
            D.rows[l] = (int32_t*)(base + F.rows[l]);
            D.wpre[l] = (uint64_t*)(base + F.wpre[l]);
        }
    }
    // one host image of keys and job tables (each table within its region)
    const size_t need[6] = {sizeof(FilterKey) * G->keys.size(), sizeof(CompactJob) * G->compact_jobs.size(),
                            sizeof(ScatterJob) * G->scatter_jobs.size(), sizeof(RefineJob) * G->refine_jobs.size(),
                            sizeof(CpiJob) * G->cpi_jobs.size(), 4 * G->first.size()};
    const size_t at[7] = {G->o_keys, G->o_cmp, G->o_sct, G->o_ref, G->o_cpi, G->o_first, G->jobs_end};
    for (int t = 0; t < 6; t++)
        if (at[t] + need[t] > at[t + 1]) {
            set_error(GFD_ERR_CUDA, "internal: job table %d needs %zu bytes, region holds %zu", t, need[t],
                      at[t + 1] - at[t]);
            return GFD_ERR_CUDA;
        }
    std::vector<uint8_t> img(G->jobs_end - G->o_jobs, 0);
    auto put = [&](size_t off, const void* p, size_t bytes) {
        if (bytes) memcpy(img.data() + (off - G->o_jobs), p, bytes);
    };
    put(G->o_keys, G->keys.data(), sizeof(FilterKey) * G->keys.size());
    put(G->o_cmp, G->compact_jobs.data(), sizeof(CompactJob) * G->compact_jobs.size());
    put(G->o_sct, G->scatter_jobs.data(), sizeof(ScatterJob) * G->scatter_jobs.size());
    put(G->o_ref, G->refine_jobs.data(), sizeof(RefineJob) * G->refine_jobs.size());
    put(G->o_cpi, G->cpi_jobs.data(), sizeof(CpiJob) * G->cpi_jobs.size());
    put(G->o_first, G->first.data(), 4 * G->first.size());
    GFD_CUDA(cudaMemcpyAsync(base + G->o_jobs, img.data(), img.size(), cudaMemcpyHostToDevice, st));
    // descriptors into the slot tables (contiguous runs in one copy) and states
    // cleared, idle (cur = -1): a serving session's running enumeration may
    // read these slots' states while they are built, and must see them idle
    // until they are started
    G->state_img.assign(n, SlotState{});
    for (auto& z : G->state_img) z.cur = -1;
    for (int s = 0; s < n;) {
        int e = s + 1;
        while (e < n && G->slot[e] == G->slot[e - 1] + 1) e++;
        GFD_CUDA(cudaMemcpyAsync(&T.desc[G->slot[s]], &G->descs[s], sizeof(SlotDesc) * (e - s),
                                 cudaMemcpyHostToDevice, st));
        GFD_CUDA(cudaMemcpyAsync(&T.state[G->slot[s]], &G->state_img[s], sizeof(SlotState) * (e - s),
                                 cudaMemcpyHostToDevice, st));
        s = e;
    }
    return GFD_OK;
}

int group_launch(gfd_graph* g, Group* G, const Tables& T, cudaMemPool_t pool, cudaStream_t st, ProfEvents& prof,
                 int64_t* launches, bool count = false) {
    const DevGraph& dg = g->dg;
    uint8_t* base = G->base;
    const ScanCount scan = count ? (ScanCount)&T.sched->cnt[CNT_SCAN_CANDS] : nullptr;
    prof.begin(PROF_FILTER, st);
    if (int rc = launch_filter(dg, (const FilterKey*)(base + G->o_keys), (int)G->keys.size(),
                               (uint32_t*)(base + G->o_keybm), st))
        return rc;
    launches[PROF_FILTER]++;
    GFD_CUDA(cudaMemsetAsync(base + G->o_zero, 0, G->o_zero_end - G->o_zero, st));
    prof.end(PROF_FILTER, st);
    prof.begin(PROF_REFINE, st);
    for (const Phase& ph : G->phases) {
        if (ph.kind == 3) {
            GFD_CUDA(cudaMemsetAsync(base + G->o_marks, 0, 4ull * dg.nwords * ph.count, st));
            continue;
        }
        const int rc = ph.kind == 2 ? launch_clear(dg, (const RefineJob*)(base + G->o_ref) + ph.first, (int)ph.count, st)
                     : ph.kind == 0 ? launch_scatter(dg, (const ScatterJob*)(base + G->o_sct) + ph.first, (int)ph.count,
                                                     ph.launch, scan, st)
                                    : launch_refine(dg, (const RefineJob*)(base + G->o_ref) + ph.first, (int)ph.count,
                                                    ph.launch, scan, st);
        if (rc) return rc;
        launches[PROF_REFINE]++;
    }
    if (int rc = launch_compact(dg, (const CompactJob*)(base + G->o_cmp), (int)G->compact_jobs.size(), st)) return rc;
    launches[PROF_REFINE] += 2;
    prof.end(PROF_REFINE, st);
    prof.begin(PROF_INDEX, st);
    const int ncpi = (int)G->cpi_jobs.size();
    if (ncpi) {
        CpiJob* d_cpi = (CpiJob*)(base + G->o_cpi);
        if (int rc = launch_cpi_count(dg, d_cpi, ncpi, G->cpi_launch, G->cpi_nch, T.err, scan, st)) return rc;
        if (!G->idx_inside) {
            // size the index edges exactly: one read-back of the per-edge totals
            std::vector<uint32_t> tot(ncpi);
            GFD_CUDA(cudaMemcpyAsync(tot.data(), base + G->o_cpi_tot, 4ull * ncpi, cudaMemcpyDeviceToHost, st));
            GFD_CUDA(cudaStreamSynchronize(st));
            std::vector<size_t> at(ncpi);
            size_t bytes = 256;
            for (int j = 0; j < ncpi; j++) {
                at[j] = bytes;
                bytes = (bytes + G->index[j].entry() * std::max<uint32_t>(1, tot[j]) + 255) & ~(size_t)255;
            }
            void* p = nullptr;
            if (int rc = pool_alloc(pool, bytes, st, &p, "index edges")) return rc;
            G->cpi_base = (uint8_t*)p;
            G->cpi_bytes = bytes;
            for (int j = 0; j < ncpi; j++) {
                G->cpi_jobs[j].idx = (int2*)(G->cpi_base + at[j]);
                G->cpi_jobs[j].cap = tot[j];
            }
            for (int s = 0; s < G->n; s++)
                for (int i = 1; i < G->plans[s].k; i++)
                    if (G->plans[s].lv[i].par >= 0) G->descs[s].cpi_idx[i] = G->cpi_jobs[G->level_index[s][i]].idx;
            GFD_CUDA(cudaMemcpyAsync(d_cpi, G->cpi_jobs.data(), sizeof(CpiJob) * ncpi, cudaMemcpyHostToDevice, st));
            // (descriptors of neighbouring slots in one copy)
            for (int s = 0; s < G->n;) {
                int e = s + 1;
                while (e < G->n && G->slot[e] == G->slot[e - 1] + 1) e++;
                GFD_CUDA(cudaMemcpyAsync(&T.desc[G->slot[s]], &G->descs[s], sizeof(SlotDesc) * (e - s),
                                         cudaMemcpyHostToDevice, st));
                s = e;
            }
        }
        if (int rc = launch_cpi_fill(dg, d_cpi, ncpi, G->cpi_launch, scan, st)) return rc;
        launches[PROF_INDEX] += 4;
    }
    prof.end(PROF_INDEX, st);
    return GFD_OK;
}

// kernel_variant 1..N selects a variant; 0 takes the graph's tuned one.
int pick_variant(const gfd_graph* g, const gfd_opts* o) {
    if (o && o->kernel_variant >= 1 && o->kernel_variant <= N_VARIANTS) return o->kernel_variant - 1;
    return g->tuned_variant >= 0 ? g->tuned_variant : 0;
}

// work items per block visit in units of the block size (1..MAX_TILE_ITERS)
int pick_tile_iters(const gfd_graph* g, const gfd_opts* o) {
    if (o && o->tile_iters >= 1) return std::min(o->tile_iters, MAX_TILE_ITERS);
    return g->tuned_tile_iters > 0 ? g->tuned_tile_iters : 8;
}

int64_t default_budget(const gfd_graph* g, const gfd_opts* o) {
    if (o && o->frontier_budget_bytes > 0) return o->frontier_budget_bytes;
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
        cudaGetLastError();
        return (int64_t)1 << 32;
    }
    // memory this graph's pool holds from earlier calls but does not use is
    // free for this one too (the pool keeps what it has allocated)
    if (g && g->eng && g->eng->pool) {
        uint64_t reserved = 0, used = 0;
        if (cudaMemPoolGetAttribute(g->eng->pool->p, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess &&
            cudaMemPoolGetAttribute(g->eng->pool->p, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess &&
            reserved > used)
            fr += (size_t)(reserved - used);
        cudaGetLastError();
    }
    // larger frontiers mean fewer, fuller steps (batched workload: 64 GiB ->
    // 542 steps, 128 GiB -> 275 steps and 5 % less time); half the free memory
    // at most
    return (int64_t)std::min<size_t>((size_t)128 << 30, fr / 2);
}

gfd_result* make_result(const gfd_graph* g, const HostPlan& P, const SlotState& S, uint64_t steps, uint64_t probes,
                        int32_t* d_viol, std::shared_ptr<DevBlock> mem, cudaStream_t st) {
    gfd_result* r = new gfd_result();
    r->k = P.k;
    r->n_matches = S.n_matches;
    r->n_viol = S.n_viol;
    r->d_viol = d_viol;
    r->mem = std::move(mem);
    r->vbits = 1;
    while (r->vbits < 32 && (1ll << r->vbits) < (int64_t)g->n) r->vbits++;
    r->stream = st;
    r->stat[0] = steps;
    r->stat[1] = S.st_work;
    r->stat[2] = S.st_rows;
    r->stat[3] = probes;
    uint64_t nc = 0;
    for (int i = 0; i < P.k; i++) nc += S.ncand[i];
    r->stat[4] = nc;
    r->stat[5] = S.st_cpi;
    return r;
}

}  // namespace

// ------------------------------------------------------------------ batch runs
int run_batch(gfd_graph* g, const gfd_gfd* const* phis, int32_t n, const gfd_opts* o, gfd_result** out, bool narrow) {
    if (!g || (!phis && n > 0) || !out || n < 0) {
        set_error(GFD_ERR_INVALID_ARG, "validate: NULL argument");
        return GFD_ERR_INVALID_ARG;
    }
    if (n == 0) return GFD_OK;
    if (n > GFD_MAX_SLOTS) {
        set_error(GFD_ERR_UNSUPPORTED, "validate: %d GFDs in one call, at most %d (split the batch)", n,
                  GFD_MAX_SLOTS);
        return GFD_ERR_UNSUPPORTED;
    }
    const int32_t flags = o ? o->flags : 0;
    const bool persistent = !(flags & GFD_FLAG_HOST_LOOP);
    const bool use_graph = !(flags & GFD_FLAG_NO_GRAPH);
    const int variant = pick_variant(g, o);
    const int block_threads = variant_threads(variant);
    cudaStream_t st = (o && o->cuda_stream) ? (cudaStream_t)o->cuda_stream : g->stream;
    const uint64_t vcap = o && o->max_violations_hint > 0 ? (uint64_t)o->max_violations_hint : (1ull << 22);

    if (g->eng && g->eng->pool) g->eng->pool->drain();
    Group G;
    const int64_t budget = (!o || o->frontier_budget_bytes <= 0) && g->tuned_budget > 0 ? g->tuned_budget
                                                                                        : default_budget(g, o);
    if (int rc = group_plan(g, phis, n, o, budget / n, &G, o && o->frontier_budget_bytes > 0, !narrow)) return rc;
    int kmax = 1;
    for (auto& P : G.plans) kmax = std::max(kmax, P.k);
    std::shared_ptr<Pool> shared_pool;
    if (int rc = get_pool(g, &shared_pool)) return rc;
    const cudaMemPool_t pool = shared_pool->p;
    Tables T;
    if (int rc = tables_alloc(pool, n, block_threads, pick_tile_iters(g, o), kmax, vcap, true, st, &T)) return rc;
    struct Free {
        std::vector<void*> p;
        cudaStream_t st;
        void now() {
            for (void* q : p)
                if (q) cudaFreeAsync(q, st);
            p.clear();
        }
        ~Free() { now(); }
    } fr{{T.base}, st};
    void* wb = nullptr;
    if (pool_alloc(pool, G.bytes, st, &wb, "device workspace")) {
        G = Group{};
        if (int rc = group_plan(g, phis, n, o, budget / n, &G, o && o->frontier_budget_bytes > 0, !narrow, Room::LEAN)) return rc;
        if (int rc = pool_alloc(pool, G.bytes, st, &wb, "device workspace")) return rc;
    }
    fr.p.push_back(wb);
    G.base = (uint8_t*)wb;
    G.slot.resize(n);
    for (int s = 0; s < n; s++) G.slot[s] = s;
    if (int rc = group_build(g, &G, T, st)) return rc;
    ProfEvents prof;
    if (int rc = prof.init((flags & GFD_FLAG_PROFILE) != 0)) return rc;
    int64_t launches[5] = {0, 0, 0, 0, 0};
    const bool count = (flags & GFD_FLAG_COUNT) != 0;
    const int lrc = group_launch(g, &G, T, pool, st, prof, launches, count);
    fr.p.push_back(G.cpi_base);
    if (lrc) return lrc;
    EnumArgs A = enum_args(g, T, kmax);
    A.narrow = narrow;
    if (G.big_bytes) {
        A.big = G.base + G.o_big;
        A.big_bytes = G.big_bytes;
    }
    if (int rc = enum_init(A, st)) return rc;
    bool general = false;  // any slot needing the general expansion
    for (int s = 0; s < n; s++) general |= G.plans[s].push_x || G.plans[s].n_components > 1;
    if (int rc = enum_run(A, persistent || count, use_graph, variant, general, st,
                          prof.on ? prof.ev[2 * PROF_ENUM] : nullptr, prof.on ? prof.ev[2 * PROF_ENUM + 1] : nullptr,
                          &launches[PROF_ENUM], count))
        return rc;
    launches[PROF_ENUM] += 1;

    std::vector<SlotState> states(n);
    Sched hs{};
    int32_t herr = 0;
    GFD_CUDA(cudaMemcpyAsync(states.data(), T.state, sizeof(SlotState) * n, cudaMemcpyDeviceToHost, st));
    GFD_CUDA(cudaMemcpyAsync(&hs, T.sched, sizeof(Sched), cudaMemcpyDeviceToHost, st));
    GFD_CUDA(cudaMemcpyAsync(&herr, T.err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    GFD_CUDA(cudaStreamSynchronize(st));
    if (hs.err == DERR_TIMEOUT) {
        set_error(GFD_ERR_TIMEOUT, "a device-side limit ran out (grid barrier wait or enumeration time)");
        return GFD_ERR_TIMEOUT;
    }
    if (herr) {
        set_error(GFD_ERR_OVERFLOW, "index capacity exceeded");
        return GFD_ERR_OVERFLOW;
    }
    bool again = false;
    for (int s = 0; s < n; s++) {
        if (states[s].err == DERR_WIDE) {
            again = true;
        } else if (states[s].err) {
            set_error(GFD_ERR_OVERFLOW, "GFD %d: partial-match counter overflow (lower chunk_rows)", s);
            return GFD_ERR_OVERFLOW;
        }
    }
    if (again) {
        // a step's partial matches without a row were more, or longer, than may be
        // expanded in place: once more with steps that always have their rows
        fr.now();
        GFD_CUDA(cudaStreamSynchronize(st));
        gfd_opts o2 = o ? *o : gfd_opts{};
        o2.cuda_stream = st;
        const int rc = run_batch(g, phis, n, &o2, out, true);
        if (rc == GFD_OK)
            for (int s = 0; s < n; s++) out[s]->stat[6] += 1;
        return rc;
    }
    if (hs.varena_used > vcap) {
        // the violations did not fit: run again with room for exactly all of them
        gfd_opts o2 = o ? *o : gfd_opts{};
        o2.max_violations_hint = (int64_t)hs.varena_used;
        o2.cuda_stream = st;
        const int rc = run_batch(g, phis, n, &o2, out, narrow);
        if (rc == GFD_OK)
            for (int s = 0; s < n; s++) out[s]->stat[6] += 1;
        return rc;
    }
    // split the arena into one violation list per GFD (order within a list is
    // arbitrary; gfd_result_tuples sorts)
    std::vector<int32_t*> vbuf(n, nullptr);
    std::vector<std::shared_ptr<DevBlock>> vmem(n);
    std::shared_ptr<Done> split;  // on another stream than the graph's
    if (hs.varena_used && st != g->stream) {
        split = std::make_shared<Done>();
        GFD_CUDA(cudaEventCreateWithFlags(&split->ev, cudaEventDisableTiming));
    }
    size_t small = 0;
    auto list_bytes = [&](int s) { return 4ull * states[s].n_viol * G.plans[s].k; };
    for (int s = 0; s < n; s++)
        if (list_bytes(s) <= SHARED_LIST) small += list_bytes(s);
    if (small) {
        void* p = nullptr;
        if (int rc = pool_alloc(pool, small, st, &p, "violation lists")) return rc;
        auto block = std::make_shared<DevBlock>(p, shared_pool, split);
        int32_t* at = (int32_t*)p;
        for (int s = 0; s < n; s++)
            if (states[s].n_viol && list_bytes(s) <= SHARED_LIST) {
                vbuf[s] = at;
                vmem[s] = block;
                at += list_bytes(s) / 4;
            }
    }
    for (int s = 0; s < n; s++) {
        if (list_bytes(s) <= SHARED_LIST) continue;
        void* p = nullptr;
        if (int rc = pool_alloc(pool, list_bytes(s), st, &p, "violation list")) return rc;
        vbuf[s] = (int32_t*)p;
        vmem[s] = std::make_shared<DevBlock>(p, shared_pool, split);
    }
    if (hs.varena_used) {
        GFD_CUDA(cudaMemcpyAsync(T.vptr, vbuf.data(), sizeof(int32_t*) * n, cudaMemcpyHostToDevice, st));
        GFD_CUDA(cudaMemsetAsync(T.vcur, 0, 8ull * n, st));
        if (int rc = launch_split(T.desc, T.varena, hs.varena_used, T.vstride, T.vptr, T.vcur, st)) return rc;
        if (split) GFD_CUDA(cudaEventRecord(split->ev, st));
        launches[PROF_ENUM] += 1;  // the split belongs to the enumeration's output
    }
    // the refined candidate lists, kept for inspection when asked for
    std::vector<std::vector<std::vector<int32_t>>> kept(n);
    if (flags & GFD_FLAG_KEEP_CANDIDATES) {
        for (int s = 0; s < n; s++) {
            kept[s].resize(G.plans[s].k);
            for (int i = 0; i < G.plans[s].k; i++) {
                auto& lst = kept[s][G.plans[s].order[i]];
                lst.resize(states[s].ncand[i]);
                if (!lst.empty())
                    GFD_CUDA(cudaMemcpyAsync(lst.data(), G.descs[s].cand[i], 4ull * lst.size(),
                                             cudaMemcpyDeviceToHost, st));
            }
        }
        std::vector<uint32_t> orig((size_t)g->n);  // lists leave in the caller's ids, increasing
        GFD_CUDA(cudaMemcpyAsync(orig.data(), g->dg.orig, 4ull * g->n, cudaMemcpyDeviceToHost, st));
        GFD_CUDA(cudaStreamSynchronize(st));
        for (auto& lists : kept)
            for (auto& lst : lists) {
                for (auto& v : lst) v = (int32_t)orig[v];
                std::sort(lst.begin(), lst.end());
            }
    }
    for (int s = 0; s < n; s++) {
        gfd_result* r = make_result(g, G.plans[s], states[s], hs.steps, hs.probes, vbuf[s], std::move(vmem[s]), st);
        if (count) {
            for (int c = 0; c < N_CNT; c++) r->stat[7 + c] = hs.cnt[c];
            // the host's figures: distinct filter keys and candidate bitmaps
            // built (for the filter and bitmap bytes)
            r->stat[7 + CNT_HOST] = ((uint64_t)G.keys.size() << 32) | (uint64_t)G.compact_jobs.size();
        }
        if (flags & GFD_FLAG_KEEP_CANDIDATES) {
            r->cand = std::move(kept[s]);
            r->has_cand = true;
        }
        for (int w = 0; w < 5; w++) {
            r->prof_ms[w] = prof.ms(w);
            r->prof_launch[w] = launches[w];
        }
        out[s] = r;
    }
    return GFD_OK;
}

// ------------------------------------------------------------------ serving
namespace {

struct Request {
    int64_t id = -1;
    // an owned copy of the GFD
    std::vector<int32_t> node_label, esrc, edst, elabel;
    std::vector<gfd_literal> X, Y;
    gfd_gfd phi{};
    void fix() {
        phi.node_label = node_label.data();
        phi.esrc = esrc.data();
        phi.edst = edst.data();
        phi.elabel = elabel.data();
        phi.X = X.data();
        phi.Y = Y.data();
    }
};

struct SlotHost {
    bool busy = false;
    bool started = false;  // its index is built and its enumeration started
    int64_t id = -1;
    std::shared_ptr<Group> group;
    int index = 0;  // position inside the group
    int32_t* viol = nullptr;
    uint64_t viol_cap = 0;
    std::unique_ptr<Request> req;
};

}  // namespace

}  // namespace gfd

struct gfd_session {
    gfd_graph* g = nullptr;
    gfd_opts opts{};
    cudaStream_t st = nullptr;        // enumeration rounds
    cudaStream_t st_admit = nullptr;  // index builds of admitted requests
    cudaEvent_t ev_admit = nullptr;   // an admission's index build is complete
    cudaEvent_t ev_round[2] = {nullptr, nullptr};  // around the rounds of a step
    gfd::SlotState* h_states = nullptr;  // pinned snapshot after a round
    gfd::Sched* h_sched = nullptr;
    int32_t* h_err = nullptr;
    std::shared_ptr<gfd::Pool> shared_pool;
    cudaMemPool_t pool = nullptr;
    gfd::Tables T;
    int variant = 0;
    int block_threads = 256;
    int64_t budget = 0;     // device bytes for the workspaces of running requests
    int64_t used = 0;
    uint64_t viol_cap = 0;  // violations stored per request before it is run again alone
    int32_t steps_per_round = 8;
    std::vector<gfd::SlotHost> slots;
    std::deque<std::unique_ptr<gfd::Request>> queue;
    std::deque<std::pair<int64_t, gfd_result*>> done;
    int64_t next_id = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    double stat[5] = {0, 0, 0, 0, 0};  // gfd_session_stat
    double admit_ms_avg = 0;  // running averages: one admission, one round
    double round_ms_avg = 0;
};

namespace gfd {

int session_create(gfd_graph* g, int32_t max_slots, const gfd_opts* o, gfd_session** out) {
    if (!g || !out || max_slots < 1 || max_slots > GFD_MAX_SLOTS) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_session_create: bad argument");
        return GFD_ERR_INVALID_ARG;
    }
    auto S = std::make_unique<gfd_session>();
    S->g = g;
    if (o) S->opts = *o;
    S->st = o && o->cuda_stream ? (cudaStream_t)o->cuda_stream : g->stream;
    S->variant = pick_variant(g, o);
    S->block_threads = variant_threads(S->variant);
    S->budget = default_budget(g, o);
    S->viol_cap = o && o->max_violations_hint > 0 ? (uint64_t)o->max_violations_hint : (1ull << 20);
    S->slots.resize(max_slots);
    // index builds run beside the enumeration rounds at the highest stream
    // priority, so their blocks are scheduled as soon as the rounds free an SM
    int prio_least = 0, prio_greatest = 0;
    GFD_CUDA(cudaDeviceGetStreamPriorityRange(&prio_least, &prio_greatest));
    GFD_CUDA(cudaStreamCreateWithPriority(&S->st_admit, cudaStreamNonBlocking, prio_greatest));
    GFD_CUDA(cudaEventCreateWithFlags(&S->ev_admit, cudaEventDisableTiming));
    GFD_CUDA(cudaEventCreate(&S->ev_round[0]));
    GFD_CUDA(cudaEventCreate(&S->ev_round[1]));
    GFD_CUDA(cudaMallocHost((void**)&S->h_states, sizeof(SlotState) * max_slots));
    GFD_CUDA(cudaMallocHost((void**)&S->h_sched, sizeof(Sched)));
    GFD_CUDA(cudaMallocHost((void**)&S->h_err, sizeof(int32_t)));
    if (int rc = get_pool(g, &S->shared_pool)) return rc;
    S->pool = S->shared_pool->p;
    if (int rc = tables_alloc(S->pool, max_slots, S->block_threads, pick_tile_iters(g, o), 0, 0, false, S->st, &S->T))
        return rc;
    if (int rc = mark_idle(S->T.state, max_slots, S->st)) return rc;  // every slot starts idle
    // the enumeration steps of one round, captured once (the tables never move)
    const EnumArgs A = enum_args(g, S->T, MAXK);  // any request
    if (int rc = capture_steps(A, S->variant, S->steps_per_round, S->st, &S->graph, &S->exec)) return rc;
    GFD_CUDA(cudaStreamSynchronize(S->st));
    *out = S.release();
    return GFD_OK;
}

void session_free(gfd_session* S) {
    if (!S) return;
    if (S->st_admit) cudaStreamSynchronize(S->st_admit);
    cudaStreamSynchronize(S->st);
    for (auto& d : S->done) gfd_result_free(d.second);
    for (auto& sl : S->slots) {
        if (sl.viol) cudaFreeAsync(sl.viol, S->st);
        if (sl.group && --sl.group->live == 0) {
            if (sl.group->base) cudaFreeAsync(sl.group->base, S->st);
            if (sl.group->cpi_base) cudaFreeAsync(sl.group->cpi_base, S->st);
        }
        sl.group.reset();
    }
    if (S->T.base) cudaFreeAsync(S->T.base, S->st);
    if (S->exec) cudaGraphExecDestroy(S->exec);
    if (S->graph) cudaGraphDestroy(S->graph);
    cudaStreamSynchronize(S->st);
    if (S->h_states) cudaFreeHost(S->h_states);
    if (S->h_sched) cudaFreeHost(S->h_sched);
    if (S->h_err) cudaFreeHost(S->h_err);
    if (S->ev_admit) cudaEventDestroy(S->ev_admit);
    for (auto e : S->ev_round)
        if (e) cudaEventDestroy(e);
    if (S->st_admit) cudaStreamDestroy(S->st_admit);
    cudaGetLastError();  // a failure here must not surface in a later, unrelated call
    delete S;
}

int session_submit(gfd_session* S, const gfd_gfd* phi, int64_t* id) {
    if (!S || !phi || !id) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_session_submit: NULL argument");
        return GFD_ERR_INVALID_ARG;
    }
    // plan now so that an invalid GFD is reported at submission
    HostPlan P;
    if (int rc = make_plan(phi, S->g->n_attrs, S->g->plan_stats(), &P, !(S->opts.flags & GFD_FLAG_NON_INDUCED),
                           (S->opts.flags & GFD_FLAG_PUSH_X) != 0))
        return rc;
    auto R = std::make_unique<Request>();
    R->id = S->next_id++;
    R->node_label.assign(phi->node_label, phi->node_label + phi->k);
    for (int e = 0; e < phi->m; e++) {
        R->esrc.push_back(phi->esrc[e]);
        R->edst.push_back(phi->edst[e]);
        R->elabel.push_back(phi->elabel[e]);
    }
    if (phi->nx) R->X.assign(phi->X, phi->X + phi->nx);
    if (!phi->y_false && phi->ny) R->Y.assign(phi->Y, phi->Y + phi->ny);
    R->phi = *phi;
    R->phi.ny = phi->y_false ? 0 : phi->ny;
    R->fix();
    *id = R->id;
    S->queue.push_back(std::move(R));
    return GFD_OK;
}

namespace {

// Admit queued requests, in arrival order, while a slot is free and their
// device memory (workspace and violation buffer) fits the budget; the admitted
// ones are planned and indexed together as one group.
int session_admit(gfd_session* S) {
    std::vector<int> free_slots;
    for (int i = 0; i < (int)S->slots.size(); i++)
        if (!S->slots[i].busy) free_slots.push_back(i);
    if (free_slots.empty() || S->queue.empty()) return GFD_OK;
    const int64_t per_slot = S->budget / (int64_t)S->slots.size();
    std::vector<std::unique_ptr<Request>> take;
    std::vector<const gfd_gfd*> phis;
    int64_t need = 0;
    while (!S->queue.empty() && take.size() < free_slots.size()) {
        Request* R = S->queue.front().get();
        Group trial;
        const gfd_gfd* one[1] = {&R->phi};
        if (int rc = group_plan(S->g, one, 1, &S->opts, per_slot, &trial, false, false, Room::SESSION)) return rc;
        const int64_t req_bytes =
            (int64_t)(trial.bytes + (trial.idx_inside ? 0 : trial.cpi_bound)) + (int64_t)(4ull * trial.plans[0].k * S->viol_cap);
        const bool idle = S->used == 0 && take.empty();  // always admit into an idle device
        if (!idle && S->used + need + req_bytes > S->budget) break;
        need += req_bytes;
        phis.push_back(&R->phi);
        take.push_back(std::move(S->queue.front()));
        S->queue.pop_front();
    }
    if (take.empty()) return GFD_OK;
    const int n = (int)take.size();
    S->stat[3] += n;
    S->stat[4] += 1;
    // the index build runs on the admission stream, beside the round that the
    // caller may have launched on the session stream
    cudaStream_t sa = S->st_admit;
    auto G = std::make_shared<Group>();
    if (int rc = group_plan(S->g, phis.data(), n, &S->opts, per_slot, G.get(), false, false, Room::SESSION)) return rc;
    void* wb = nullptr;
    if (int rc = pool_alloc(S->pool, G->bytes, sa, &wb, "request workspace")) return rc;
    G->base = (uint8_t*)wb;
    G->slot.assign(free_slots.begin(), free_slots.begin() + n);
    S->used += (int64_t)G->bytes;
    for (int i = 0; i < n; i++) {
        void* vp = nullptr;
        if (int rc = pool_alloc(S->pool, 4ull * G->plans[i].k * S->viol_cap, sa, &vp, "violation buffer")) return rc;
        G->descs[i].viol = (int32_t*)vp;
        G->descs[i].viol_cap = S->viol_cap;
        S->used += (int64_t)(4ull * G->plans[i].k * S->viol_cap);
        SlotHost& sl = S->slots[G->slot[i]];
        sl.busy = true;
        sl.id = take[i]->id;
        sl.group = G;
        sl.index = i;
        sl.viol = (int32_t*)vp;
        sl.viol_cap = S->viol_cap;
        sl.req = std::move(take[i]);
    }
    G->live = n;
    if (int rc = group_build(S->g, G.get(), S->T, sa)) return rc;
    ProfEvents prof;
    int64_t launches[5] = {0, 0, 0, 0, 0};
    const int lrc = group_launch(S->g, G.get(), S->T, S->pool, sa, prof, launches);
    S->used += (int64_t)G->cpi_bytes;
    if (lrc) return lrc;
    // the session stream starts the new slots once their index is built (after
    // whatever round it is running)
    GFD_CUDA(cudaEventRecord(S->ev_admit, sa));
    GFD_CUDA(cudaStreamWaitEvent(S->st, S->ev_admit, 0));
    if (int rc = init_slots(enum_args(S->g, S->T, MAXK), G->slot.data(), n, S->st)) return rc;
    for (int i = 0; i < n; i++) S->slots[G->slot[i]].started = true;
    return GFD_OK;
}

}  // namespace

namespace {

// Free a slot's device memory and return it to the pool of free slots (its
// request finished or was cancelled; no kernel of the session is running).
void slot_release(gfd_session* S, SlotHost& sl) {
    if (sl.viol) cudaFreeAsync(sl.viol, S->st);
    sl.viol = nullptr;
    S->used -= (int64_t)(4ull * sl.group->plans[sl.index].k * sl.viol_cap);
    if (--sl.group->live == 0) {
        cudaFreeAsync(sl.group->base, S->st);
        if (sl.group->cpi_base) cudaFreeAsync(sl.group->cpi_base, S->st);
        S->used -= (int64_t)(sl.group->bytes + sl.group->cpi_bytes);
        sl.group->base = nullptr;
        sl.group->cpi_base = nullptr;
    }
    sl.group.reset();
    sl.req.reset();
    sl.busy = false;
    sl.started = false;
    sl.id = -1;
}

}  // namespace

int session_step(gfd_session* S, int32_t* n_advanced, int32_t* n_running, int32_t* n_queued) {
    if (!S) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_session_step: NULL session");
        return GFD_ERR_INVALID_ARG;
    }
    using clk = std::chrono::steady_clock;
    // The round for the requests already running is launched first, its state
    // snapshot copied to pinned memory behind it; queued requests are admitted
    // meanwhile (planning on the host, index build on the admission stream), so
    // admission overlaps the round; the new requests start after it.
    std::vector<char> in_round(S->slots.size(), 0);
    int busy = 0;  // requests in the round
    // while an admission keeps the host busy, the GPU should not run dry: queue
    // as many rounds as the last admissions took, by the running averages
    const bool admitting = !S->queue.empty();
    int rounds = 1;
    if (admitting && S->round_ms_avg > 0)
        rounds = (int)std::min(16.0, std::max(1.0, std::ceil(S->admit_ms_avg / S->round_ms_avg)));
    int launched = 0;
    auto launch_round = [&]() -> int {
        busy = 0;
        for (size_t i = 0; i < S->slots.size(); i++) {
            in_round[i] = S->slots[i].busy && S->slots[i].started;
            busy += in_round[i];
        }
        if (!busy) return GFD_OK;
        GFD_CUDA(cudaEventRecord(S->ev_round[0], S->st));
        for (int r = 0; r < rounds; r++) GFD_CUDA(cudaGraphLaunch(S->exec, S->st));
        GFD_CUDA(cudaEventRecord(S->ev_round[1], S->st));
        launched = rounds;
        GFD_CUDA(cudaMemcpyAsync(S->h_states, S->T.state, sizeof(SlotState) * S->slots.size(),
                                 cudaMemcpyDeviceToHost, S->st));
        GFD_CUDA(cudaMemcpyAsync(S->h_sched, S->T.sched, sizeof(Sched), cudaMemcpyDeviceToHost, S->st));
        GFD_CUDA(cudaMemcpyAsync(S->h_err, S->T.err, sizeof(int32_t), cudaMemcpyDeviceToHost, S->st));
        return GFD_OK;
    };
    const auto t0 = clk::now();
    if (int rc = launch_round()) return rc;
    const auto ta = clk::now();
    const int64_t admissions_before = (int64_t)S->stat[4];
    if (int rc = session_admit(S)) return rc;
    const auto t1 = clk::now();
    const double admit_ms = std::chrono::duration<double, std::milli>(t1 - ta).count();
    S->stat[0] += admit_ms;
    if ((int64_t)S->stat[4] > admissions_before)
        S->admit_ms_avg = S->admit_ms_avg > 0 ? 0.8 * S->admit_ms_avg + 0.2 * admit_ms : admit_ms;
    if (!busy) {
        rounds = 1;
        if (int rc = launch_round()) return rc;  // nothing was running: run the admitted requests now
    }
    if (n_advanced) *n_advanced = busy;
    if (busy) {
        GFD_CUDA(cudaStreamSynchronize(S->st));
        float gpu_ms = 0;  // the rounds' device time (they may overlap an admission)
        if (cudaEventElapsedTime(&gpu_ms, S->ev_round[0], S->ev_round[1]) != cudaSuccess) {
            cudaGetLastError();
            gpu_ms = 0;
        }
        S->stat[1] += gpu_ms;
        S->stat[2] += launched;
        if (gpu_ms > 0) {
            const double per = gpu_ms / launched;
            S->round_ms_avg = S->round_ms_avg > 0 ? 0.8 * S->round_ms_avg + 0.2 * per : per;
        }
        const SlotState* states = S->h_states;
        const Sched& hs = *S->h_sched;
        if (hs.err == DERR_TIMEOUT) {
            set_error(GFD_ERR_TIMEOUT, "a device-side limit ran out in the serving session");
            return GFD_ERR_TIMEOUT;
        }
        if (*S->h_err) {
            set_error(GFD_ERR_OVERFLOW, "index capacity exceeded");
            return GFD_ERR_OVERFLOW;
        }
        for (size_t i = 0; i < S->slots.size(); i++) {
            SlotHost& sl = S->slots[i];
            // slots started after the round's snapshot are not in it
            if (!in_round[i] || !sl.busy || states[i].cur >= 0) continue;
            if (states[i].err && states[i].err != DERR_WIDE) {
                set_error(GFD_ERR_OVERFLOW, "request %lld: partial-match counter overflow", (long long)sl.id);
                return GFD_ERR_OVERFLOW;
            }
            gfd_result* r = nullptr;
            if (states[i].err == DERR_WIDE || states[i].n_viol > sl.viol_cap) {
                // a wide step did not come out, or there are more violations than the
                // request's buffer holds: validate it again alone
                gfd_opts o2 = S->opts;
                o2.cuda_stream = S->st;
                o2.flags &= ~GFD_FLAG_HOST_LOOP;
                o2.max_violations_hint = (int64_t)std::max(states[i].n_viol, sl.viol_cap);
                const gfd_gfd* one[1] = {&sl.req->phi};
                if (int rc = run_batch(S->g, one, 1, &o2, &r, states[i].err == DERR_WIDE)) return rc;
                r->stat[6] += 1;
                cudaFreeAsync(sl.viol, S->st);
            } else {
                r = make_result(S->g, sl.group->plans[sl.index], states[i], hs.steps, hs.probes, sl.viol,
                                std::make_shared<DevBlock>(sl.viol, S->shared_pool), S->st);
            }
            sl.viol = nullptr;  // now owned by the result (or freed above)
            S->done.emplace_back(sl.id, r);
            slot_release(S, sl);
        }
    }
    int running = 0;
    for (auto& sl : S->slots) running += sl.busy;
    if (n_running) *n_running = running;
    if (n_queued) *n_queued = (int32_t)S->queue.size();
    return GFD_OK;
}

int session_cancel(gfd_session* S, int64_t id) {
    if (!S) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_session_cancel: NULL session");
        return GFD_ERR_INVALID_ARG;
    }
    for (auto it = S->queue.begin(); it != S->queue.end(); ++it)
        if ((*it)->id == id) {
            S->queue.erase(it);
            return GFD_OK;
        }
    for (size_t i = 0; i < S->slots.size(); i++) {
        SlotHost& sl = S->slots[i];
        if (!sl.busy || sl.id != id) continue;
        // the slot stops: the next control step skips it (stream-ordered after
        // the last round, which has finished when gfd_session_step returned)
        static const int32_t stopped = -1;
        GFD_CUDA(cudaMemcpyAsync(&S->T.state[i].cur, &stopped, sizeof(int32_t), cudaMemcpyHostToDevice, S->st));
        slot_release(S, sl);
        return GFD_OK;
    }
    for (auto it = S->done.begin(); it != S->done.end(); ++it)
        if (it->first == id) {
            gfd_result_free(it->second);
            S->done.erase(it);
            return GFD_OK;
        }
    set_error(GFD_ERR_INVALID_ARG, "gfd_session_cancel: no request %lld in the session", (long long)id);
    return GFD_ERR_INVALID_ARG;
}

double session_stat(const gfd_session* S, int32_t which) {
    return S && which >= 0 && which < 5 ? S->stat[which] : 0.0;
}

int session_next_result(gfd_session* S, int64_t* id, gfd_result** out) {
    if (!S || !id || !out) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_session_next_result: NULL argument");
        return GFD_ERR_INVALID_ARG;
    }
    if (S->done.empty()) {
        *id = -1;
        *out = nullptr;
        return GFD_OK;
    }
    *id = S->done.front().first;
    *out = S->done.front().second;
    S->done.pop_front();
    return GFD_OK;
}

// ------------------------------------------------------------------ autotuner
int autotune(gfd_graph* g, const gfd_gfd* const* phis, int32_t n, const gfd_opts* o, gfd_opts* best) {
    if (!g || (!phis && n > 0) || n <= 0) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_autotune: empty batch");
        return GFD_ERR_INVALID_ARG;
    }
    const int64_t b0 = default_budget(g, o);
    const int64_t budgets[2] = {b0, std::max<int64_t>(b0 / 4, (int64_t)1 << 28)};
    const int tiles[2] = {8, 32};
    double best_ms = -1;
    int best_v = 0, best_t = 8;
    int64_t best_b = b0;
    std::vector<gfd_result*> res(n, nullptr);
    for (int bi = 0; bi < 2; bi++)
        for (int ti = 0; ti < 2; ti++)
        for (int v = 0; v < N_VARIANTS; v++) {
            gfd_opts t = o ? *o : gfd_opts{};
            t.kernel_variant = v + 1;
            t.tile_iters = tiles[ti];
            t.frontier_budget_bytes = budgets[bi];
            t.flags |= GFD_FLAG_PROFILE;
            t.flags &= ~GFD_FLAG_HOST_LOOP;
            const int rc = run_batch(g, phis, n, &t, res.data());
            if (rc == GFD_ERR_CUDA || rc == GFD_ERR_OUT_OF_MEMORY) continue;  // variant not usable here
            if (rc) return rc;
            double ms = 0;
            for (int w = 0; w < 4; w++) ms += res[0]->prof_ms[w];
            for (auto& r : res) {
                gfd_result_free(r);
                r = nullptr;
            }
            if (best_ms < 0 || ms < best_ms) {
                best_ms = ms;
                best_v = v;
                best_t = tiles[ti];
                best_b = budgets[bi];
            }
        }
    if (best_ms < 0) {
        set_error(GFD_ERR_CUDA, "gfd_autotune: no variant ran");
        return GFD_ERR_CUDA;
    }
    g->tuned_variant = best_v;
    g->tuned_tile_iters = best_t;
    g->tuned_budget = best_b;
    if (best) {
        *best = o ? *o : gfd_opts{};
        best->kernel_variant = best_v + 1;
        best->tile_iters = best_t;
        best->frontier_budget_bytes = best_b;
    }
    return GFD_OK;
}

// ------------------------------------------------------------------ result sort
namespace {

// Where a result's tuples are and go.
struct PackSrc {
    const int32_t* p;   // the result's unsorted tuples
    int32_t k;
    int32_t pad;
    uint64_t row_off;   // first row of the result (in the rows of all results, and in sorted order)
    uint64_t int_off;   // first int of the result in the packed output
};

// the result whose rows hold row g (src[nres].row_off = all rows)
__device__ __forceinline__ int src_of(const PackSrc* src, int nres, uint64_t g) {
    int lo = 0, hi = nres;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (src[mid].row_off <= g) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Short lists: a warp per tuple counts the tuples of its result that come before
// it (tuples of a result differ, so the count is its place) and writes it there.
// One launch instead of the 20 or more of a radix sort: 400 tuples of 3 take 5 us
// (the whole fetch on 20k vertices: 250 -> 32 us, with scratch from the graph's pool).
__global__ void __launch_bounds__(256) k_rank_rows(const PackSrc* src, PackSrc one, int nres, uint64_t total,
                                                   int32_t* out) {
    const int lane = threadIdx.x & 31;
    for (uint64_t g = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; g < total;
         g += ((uint64_t)gridDim.x * blockDim.x) >> 5) {
        PackSrc s = one;
        uint64_t end = total;
        if (src) {
            const int i = src_of(src, nres, g);
            s = src[i];
            end = src[i + 1].row_off;
        }
        const int k = s.k;
        const int32_t* const mine = s.p + (g - s.row_off) * k;
        const int32_t first = mine[0];
        const uint32_t rows = (uint32_t)(end - s.row_off);
        uint32_t before = 0;
        for (uint32_t j = lane; j < rows; j += 32) {
            const int32_t* const row = s.p + (uint64_t)j * k;
            const int32_t a = row[0];
            if (a != first) {
                before += a < first;
            } else {
                int c = 1;
                while (c < k && row[c] == mine[c]) c++;
                before += c < k && row[c] < mine[c];
            }
        }
        before = __reduce_add_sync(0xffffffffu, before);
        if (lane < k) out[s.int_off + (uint64_t)before * k + lane] = mine[lane];
    }
}
// Pairs of tuples compared at most (the sum of the results' squared counts):
// 2^26 pairs take 60 us, about what a radix sort takes at its smallest.
constexpr uint64_t RANK_PAIRS = 1ull << 26;

__global__ void k_iota(uint32_t* p, uint64_t n) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        p[i] = (uint32_t)i;
}

// Long lists: least-significant-first stable radix sorts of a carried permutation.
// The sort key of a row is the bit string of its columns, most significant first:
// the result's number (rbits), then k ids of vbits each; a pass sorts bits
// [b0, b0 + 64) of it, so that no pass is spent on bits that no id has.
__global__ void k_gather_key(const int32_t* t, int W, int rbits, int vbits, const uint32_t* perm, uint64_t n, int b0,
                             uint64_t* key) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const int32_t* row = t + (uint64_t)perm[i] * W;
        uint64_t x = 0;
        int at = -b0;  // position of the column's lowest bit in the key
        for (int c = W - 1; c >= 0 && at < 64; c--) {
            const int bits = c == 0 && rbits >= 0 ? rbits : vbits;
            const uint64_t v = (uint32_t)row[c];
            if (at + bits > 0) x |= at >= 0 ? v << at : v >> -at;
            at += bits;
        }
        key[i] = x;
    }
}

__global__ void k_gather_rows(const int32_t* t, int k, const uint32_t* perm, uint64_t n, int32_t* out) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n * k; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t r = i / k, c = i % k;
        out[i] = t[(uint64_t)perm[r] * k + c];
    }
}

// Several results' violation lists sorted together: rows of a matrix of
// width W = 1 + max k, column 0 the result's index (most significant), the
// tuple after it (zero-padded; only rows of the same result are ever compared
// past column 0).
__global__ void k_pack_multi(const PackSrc* src, int nres, uint64_t total, int W, int32_t* M) {
    for (uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; g < total; g += (uint64_t)gridDim.x * blockDim.x) {
        const int i = src_of(src, nres, g);
        const PackSrc s = src[i];
        const uint64_t local = g - s.row_off;
        int32_t* row = M + g * W;
        row[0] = i;
        for (int c = 0; c < W - 1; c++) row[1 + c] = c < s.k ? s.p[local * s.k + c] : 0;
    }
}

__global__ void k_unpack_multi(const PackSrc* src, const int32_t* M, int W, const uint32_t* perm, uint64_t total,
                               int32_t* out) {
    for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < total; p += (uint64_t)gridDim.x * blockDim.x) {
        const int32_t* row = M + (uint64_t)perm[p] * W;
        const PackSrc s = src[row[0]];
        int32_t* dst = out + s.int_off + (p - s.row_off) * s.k;
        for (int c = 0; c < s.k; c++) dst[c] = row[1 + c];
    }
}

// Scratch of a sort: one allocation of the result's pool, which takes it from what it
// holds unused. If the pool had to grow by more than SORT_KEEP for it, it shrinks again
// afterwards (by itself it gives nothing back before the graph is freed).
constexpr size_t SORT_KEEP = (size_t)64 << 20;
struct SortScratch {
    Layout L;
    uint8_t* base = nullptr;
    cudaStream_t st;
    std::shared_ptr<Pool> pool;
    uint64_t reserved = 0;  // what the pool held before
    explicit SortScratch(cudaStream_t s) : st(s) { L.size = 0; }
    static uint64_t held(cudaMemPool_t p) {
        uint64_t x = 0;
        if (cudaMemPoolGetAttribute(p, cudaMemPoolAttrReservedMemCurrent, &x) != cudaSuccess) cudaGetLastError();
        return x;
    }
    int alloc(const gfd_result* r) {
        void* p = nullptr;
        pool = r->mem->pool;
        if (L.size > SORT_KEEP) reserved = held(pool->p);
        if (int rc = pool_alloc(pool->p, L.size, st, &p, "violation sort")) return rc;
        base = (uint8_t*)p;
        return GFD_OK;
    }
    ~SortScratch() {
        if (!base) return;
        cudaFreeAsync(base, st);
        if (L.size > SORT_KEEP && held(pool->p) > reserved + SORT_KEEP) {
            cudaStreamSynchronize(st);
            cudaMemPoolTrimTo(pool->p, reserved);
        }
        cudaGetLastError();
    }
};

// Permutation that sorts the n rows of t (width W, `bits` key bits in all, rbits
// of column 0 or -1 when it is an id like the others).
struct RadixRows {
    size_t o_p0, o_p1, o_k0, o_k1, o_tmp, tmp_bytes = 0;
    int plan(uint64_t n, SortScratch* S) {
        cub::DoubleBuffer<uint64_t> kb(nullptr, nullptr);
        cub::DoubleBuffer<uint32_t> pb(nullptr, nullptr);
        GFD_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, kb, pb, (int64_t)n, 0, 64, S->st));
        o_p0 = S->L.take(4 * n);
        o_p1 = S->L.take(4 * n);
        o_k0 = S->L.take(8 * n);
        o_k1 = S->L.take(8 * n);
        o_tmp = S->L.take(tmp_bytes);
        return GFD_OK;
    }
    int sort(const int32_t* t, int W, int rbits, int vbits, uint64_t n, int grid, const SortScratch& S, uint32_t** perm) {
        cub::DoubleBuffer<uint64_t> kb((uint64_t*)(S.base + o_k0), (uint64_t*)(S.base + o_k1));
        cub::DoubleBuffer<uint32_t> pb((uint32_t*)(S.base + o_p0), (uint32_t*)(S.base + o_p1));
        k_iota<<<grid, 256, 0, S.st>>>(pb.Current(), n);
        const int bits = rbits >= 0 ? rbits + (W - 1) * vbits : W * vbits;
        for (int b0 = 0; b0 < bits; b0 += 64) {
            k_gather_key<<<grid, 256, 0, S.st>>>(t, W, rbits, vbits, pb.Current(), n, b0, kb.Current());
            GFD_CUDA(cub::DeviceRadixSort::SortPairs(S.base + o_tmp, tmp_bytes, kb, pb, (int64_t)n, 0,
                                                     std::min(64, bits - b0), S.st));
        }
        *perm = pb.Current();
        return GFD_OK;
    }
};

int rows_grid(uint64_t n) { return (int)std::min<uint64_t>((n + 255) / 256, (uint64_t)device_sms() * 16); }
int rank_grid(uint64_t n) { return (int)std::min<uint64_t>((n + 7) / 8, (uint64_t)device_sms() * 8); }

}  // namespace

// Device-to-host copy of results into caller memory, synchronous. (A staged
// copy through a page-locked double buffer, several host threads moving each
// chunk into pageable memory, was slower here: 67 vs 44 ms for 853 MB.)
int copy_to_host(void* dst, const void* src, size_t bytes, cudaStream_t st) {
    if (bytes == 0) return GFD_OK;
    GFD_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st));
    GFD_CUDA(cudaStreamSynchronize(st));
    return GFD_OK;
}

// Lexicographic order of the violation tuples (Vio is a set; this fixes a
// canonical order).
int result_fetch(gfd_result* r) {
    if (r->fetched) return GFD_OK;
    const uint64_t n = r->n_viol;
    if (n > 0) {
        r->tuples.reset(new (std::nothrow) int32_t[n * r->k]);
        if (!r->tuples) {
            set_error(GFD_ERR_OUT_OF_MEMORY, "violation tuples: %llu host bytes", (unsigned long long)(4ull * n * r->k));
            return GFD_ERR_OUT_OF_MEMORY;
        }
        if (int rc = result_sort_copy(r, r->tuples.get())) {
            r->tuples.reset();
            return rc;
        }
    }
    r->fetched = true;
    return GFD_OK;
}

int result_sort_copy(gfd_result* r, int32_t* dst) {
    const uint64_t n = r->n_viol;
    const int k = r->k;
    if (n == 0) return GFD_OK;
    cudaStream_t st = r->stream;
    SortScratch S(st);
    const bool rank = n <= RANK_PAIRS / n;
    RadixRows R;
    if (!rank)
        if (int rc = R.plan(n, &S)) return rc;
    const size_t o_out = S.L.take(4 * n * k);
    if (int rc = S.alloc(r)) return rc;
    int32_t* sorted = (int32_t*)(S.base + o_out);
    if (rank) {
        k_rank_rows<<<rank_grid(n), 256, 0, st>>>(nullptr, PackSrc{r->d_viol, k, 0, 0, 0}, 1, n, sorted);
    } else {
        uint32_t* perm = nullptr;
        if (int rc = R.sort(r->d_viol, k, -1, r->vbits, n, rows_grid(n), S, &perm)) return rc;
        k_gather_rows<<<rows_grid(n), 256, 0, st>>>(r->d_viol, k, perm, n, sorted);
    }
    GFD_CUDA(cudaGetLastError());
    if (int rc = copy_to_host(dst, sorted, 4 * n * k, st)) return rc;
    r->mem->written = true;
    return GFD_OK;
}

int results_sort_copy(gfd_result* const* rs, int n, int32_t* out, uint64_t capacity) {
    std::vector<PackSrc> src((size_t)n + 1);
    uint64_t total = 0, ints = 0, pairs = 0;
    int kmax = 1, vbits = 1;
    cudaStream_t st = nullptr;
    const gfd_result* any = nullptr;
    for (int r = 0; r < n; r++) {
        src[r] = PackSrc{rs[r]->d_viol, rs[r]->k, 0, total, ints};
        total += rs[r]->n_viol;
        ints += rs[r]->n_viol * (uint64_t)rs[r]->k;
        kmax = std::max(kmax, rs[r]->k);
        vbits = std::max(vbits, rs[r]->vbits);
        pairs += rs[r]->n_viol < RANK_PAIRS ? rs[r]->n_viol * rs[r]->n_viol : RANK_PAIRS + 1;
        pairs = std::min(pairs, RANK_PAIRS + 1);
        if (rs[r]->n_viol && !any) any = rs[r];
    }
    src[n] = PackSrc{nullptr, 1, 0, total, ints};
    if (capacity < ints) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_results_copy_tuples: capacity %llu < %llu ints",
                  (unsigned long long)capacity, (unsigned long long)ints);
        return GFD_ERR_INVALID_ARG;
    }
    if (total == 0) return GFD_OK;
    st = any->stream;
    // Each result's violation list is written on the stream of the call that
    // made it (the split runs after that call returns). The sort runs on the
    // first such stream, so it first waits for every other one.
    std::vector<cudaStream_t> waited;
    for (int r = 0; r < n; r++) {
        const cudaStream_t rs_st = rs[r]->stream;
        if (!rs[r]->n_viol || rs_st == st || std::find(waited.begin(), waited.end(), rs_st) != waited.end())
            continue;
        waited.push_back(rs_st);
        cudaEvent_t ev = nullptr;
        GFD_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        cudaError_t e = cudaEventRecord(ev, rs_st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev, 0);
        cudaEventDestroy(ev);
        if (e != cudaSuccess) return cuda_fail(e, "ordering the violation sort after the result's stream");
    }
    if (total >= ((uint64_t)1 << 32)) {  // the carried permutation is 32-bit: one result at a time
        for (int r = 0; r < n; r++)
            if (int rc = result_sort_copy(rs[r], out + src[r].int_off)) return rc;
        return GFD_OK;
    }
    SortScratch S(st);
    const size_t o_src = S.L.take(sizeof(PackSrc) * ((size_t)n + 1)), o_out = S.L.take(4 * ints);
    const bool rank = pairs <= RANK_PAIRS;
    const int W = kmax + 1;
    RadixRows R;
    size_t o_M = 0;
    if (!rank) {
        if (int rc = R.plan(total, &S)) return rc;
        o_M = S.L.take(4ull * total * W);
    }
    if (int rc = S.alloc(any)) return rc;
    PackSrc* d_src = (PackSrc*)(S.base + o_src);
    int32_t* dout = (int32_t*)(S.base + o_out);
    GFD_CUDA(cudaMemcpyAsync(d_src, src.data(), sizeof(PackSrc) * ((size_t)n + 1), cudaMemcpyHostToDevice, st));
    if (rank) {
        k_rank_rows<<<rank_grid(total), 256, 0, st>>>(d_src, PackSrc{}, n, total, dout);
    } else {
        int32_t* M = (int32_t*)(S.base + o_M);
        const int grid = rows_grid(total);
        int rbits = 0;
        while ((1ll << rbits) < n) rbits++;
        k_pack_multi<<<grid, 256, 0, st>>>(d_src, n, total, W, M);
        uint32_t* perm = nullptr;
        if (int rc = R.sort(M, W, rbits, vbits, total, grid, S, &perm)) return rc;
        k_unpack_multi<<<grid, 256, 0, st>>>(d_src, M, W, perm, total, dout);
    }
    GFD_CUDA(cudaGetLastError());
    if (int rc = copy_to_host(out, dout, 4 * ints, st)) return rc;
    for (int r = 0; r < n; r++)
        if (rs[r]->mem) rs[r]->mem->written = true;
    return GFD_OK;
}

}  // namespace gfd
