// gfd_graph_load / gfd_graph_free: make G = (V, E, L, F_A) (Section II)
// resident on the device.
//
// The caller's int64/int32 CSR is checked on the device (rows strictly
// increasing, ids in range, labels in range, reverse CSR equal to the transpose
// of the forward one) and packed into the layout of common.cuh. Vertices are
// renumbered inside: by degree class (hubs first), then by label, then by falling
// degree, then by id. So the scans of a candidate list know where its hubs end without
// looking at degrees (and give each class its own share of work), candidates of one
// label have adjacency lists next to each other, and the vertices that edges lead to
// most often share a few cache lines. Ids leave the library through orig[].
#include <cub/cub.cuh>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "engine.h"

namespace gfd {

namespace {

// error bits written by the validation kernels
enum : uint32_t {
    BAD_OFFSETS = 1u,
    BAD_ORDER = 2u,
    BAD_RANGE = 4u,
    BAD_LABEL = 8u,
    BAD_REVERSE = 16u,
};

__global__ void k_check_offsets(const int64_t* off, int32_t n, int64_t m, uint32_t* bad) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v <= n;
         v += (int64_t)gridDim.x * blockDim.x) {
        int64_t o = off[v];
        bool ok = o >= 0 && o <= m;
        if (v == 0) ok = ok && o == 0;
        if (v == n) ok = ok && o == m;
        if (v > 0) ok = ok && off[v - 1] <= o;
        if (!ok) atomicOr(bad, BAD_OFFSETS);
    }
}

// Largest edge label, and the number of edges of each label 0..255.
__global__ void k_edge_labels(const int32_t* lab, int64_t m, int32_t* maxlab, unsigned long long* hist) {
    __shared__ uint32_t h[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0;
    __syncthreads();
    int32_t mx = INT32_MIN;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t l = lab[e];
        mx = max(mx, l);
        if (l >= 0 && l < 256) atomicAdd(&h[l], 1u);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(maxlab, mx);
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], (unsigned long long)h[i]);
}

// One warp per row: check order / range / label; in-degrees and self-loop labels
// (label + 1, 0 none).
__global__ void k_check_rows(const int64_t* off, const int32_t* nbr, const int32_t* lab, int32_t n, int32_t lbits,
                             uint32_t* din, uint32_t* self, uint32_t* bad) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = warp; v < n; v += nwarps) {
        const int64_t a = off[v], b = off[v + 1];
        uint32_t err = 0;
        for (int64_t e = a + lane; e < b; e += 32) {
            const int32_t x = nbr[e];
            const int32_t l = lab[e];
            if (l < 0 || l > 255 || (l >> lbits) != 0) err |= BAD_LABEL;
            if (e > a && nbr[e - 1] >= x) err |= BAD_ORDER;
            if (x < 0 || x >= n) {
                err |= BAD_RANGE;
                continue;
            }
            if (din) atomicAdd(&din[x], 1u);
            if (self && x == v) self[v] = (uint32_t)(l & 255) + 1;
        }
        err = __reduce_or_sync(0xffffffffu, err);
        if (lane == 0 && err) atomicOr(bad, err);
    }
}

// Vertex info in the caller's order (label, self-loop), 32-bit offsets, and the
// key that orders the vertices inside: degree class, label, falling degree (ties
// keep the caller's order: the sort is stable).
constexpr int KEY_BITS = 2 + 16 + 32;
__global__ void k_vertex_keys(const int32_t* vlabel, const int64_t* off, const uint32_t* din, const uint32_t* self,
                              int32_t n, uint32_t* o_vinfo, uint32_t* o_out_off, uint64_t* key, uint32_t* id,
                              uint32_t* bad) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t L = vlabel[v];
        if (L < 0 || L > 65534) atomicOr(bad, BAD_LABEL);
        o_vinfo[v] = ((uint32_t)L & 0xffffu) | (self[v] << 16);
        o_out_off[v] = (uint32_t)off[v];
        const uint64_t deg = min((uint64_t)(off[v + 1] - off[v]) + din[v], (uint64_t)0xffffffffu);
        uint64_t cls = 0;
        while (cls < N_CLASS - 1 && deg <= class_degree((int)cls)) cls++;
        key[v] = (cls << 48) | ((uint64_t)((uint32_t)L & 0xffffu) << 32) | (0xffffffffull - deg);
        id[v] = (uint32_t)v;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) o_out_off[n] = (uint32_t)off[n];
}

// A maximal range of vertices of one degree class and label.
struct Segment {
    uint32_t first, label;
};

// Inside vertex i is the caller's orig[i] (key: its sort key): ranks, vertex info
// and degrees in the inside order, where the segments start (in any order), and
// where the classes end (0 where all up to a class are empty).
__global__ void k_renumber(const uint32_t* orig, const uint64_t* key, const uint32_t* o_vinfo, const int64_t* off,
                           const uint32_t* din, int32_t n, uint32_t* rank, uint32_t* vinfo, uint32_t* dout_new,
                           uint32_t* din_new, Segment* segs, uint32_t* nsegs, uint32_t* class_end) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t v = orig[i], vi = o_vinfo[v];
        rank[v] = (uint32_t)i;
        vinfo[i] = vi;
        dout_new[i] = (uint32_t)(off[v + 1] - off[v]);
        din_new[i] = din[v];
        const uint64_t cl = key[i] >> 32;
        if (i == 0 || key[i - 1] >> 32 != cl) segs[atomicAdd(nsegs, 1u)] = Segment{(uint32_t)i, vi & 0xffffu};
        // the last vertex up to each class
        const uint64_t next = i + 1 < n ? key[i + 1] >> 48 : N_CLASS;
        for (uint64_t c = cl >> 16; c < N_CLASS - 1 && c < next; c++) class_end[c] = (uint32_t)i + 1;
    }
}

__global__ void k_gather_attrs(const int32_t* src, const uint32_t* orig, int32_t n, int32_t n_attrs, int32_t* dst) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        for (int a = 0; a < n_attrs; a++) dst[(int64_t)a * n + i] = src[(int64_t)a * n + orig[i]];
}

// Sort keys of the edges of the caller's rows (renumbered by rank when given):
// (source << nb) | destination, or the reverse; labels alongside.
__global__ void k_edge_keys(const int64_t* off, const int32_t* nbr, const int32_t* lab, const uint32_t* rank, int32_t n,
                            int32_t nb, bool reverse, uint64_t* keys, uint8_t* labs) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = warp; v < n; v += nwarps) {
        const uint64_t a = rank ? rank[v] : (uint32_t)v;
        for (int64_t e = off[v] + lane; e < off[v + 1]; e += 32) {
            const uint64_t b = rank ? rank[nbr[e]] : (uint32_t)nbr[e];
            keys[e] = reverse ? (b << nb) | a : (a << nb) | b;
            labs[e] = (uint8_t)lab[e];
        }
    }
}

__global__ void k_pack_adj(const uint64_t* keys, const uint8_t* labs, int64_t m, int32_t nb, int32_t lbits, uint32_t* adj) {
    const uint64_t mask = (1ull << nb) - 1;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        adj[e] = ((uint32_t)(keys[e] & mask) << lbits) | labs[e];
}

// The caller's reverse CSR against the sorted transpose keys.
__global__ void k_compare_reverse(const int64_t* in_off, const int32_t* src, const int32_t* lab, int32_t n, int32_t nb,
                                  const uint32_t* o_in_off, const uint64_t* keys, const uint8_t* labs, uint32_t* bad) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = warp; v < n; v += nwarps) {
        const int64_t a = in_off[v], b = in_off[v + 1];
        bool differs = a != (int64_t)o_in_off[v];
        for (int64_t e = a + lane; e < b; e += 32)
            differs |= keys[e] != (((uint64_t)v << nb) | (uint32_t)src[e]) || (int32_t)labs[e] != lab[e];
        if (differs) atomicOr(bad, BAD_REVERSE);
    }
}

// One warp per vertex: OR of the signature bits of its out-neighbours (half 0)
// or in-neighbours (half 1).
__global__ void k_signature(const uint32_t* off, const uint32_t* adj, int32_t n, int32_t lbits, int half,
                            unsigned long long* sig) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = warp; v < n; v += nwarps) {
        unsigned long long b = 0;
        for (uint32_t e = off[v] + lane; e < off[v + 1]; e += 32) b |= 1ull << sig_bit(adj[e] >> lbits);
        const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)b);
        const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(b >> 32));
        if (lane == 0) sig[2 * v + half] = ((unsigned long long)hi << 32) | lo;
    }
}

// One warp per vertex: the row filter of its list (words zeroed before).
__global__ void k_row_filter(const uint32_t* off, const uint32_t* adj, int32_t n, int32_t lbits, uint32_t* filter) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = warp; v < n; v += nwarps) {
        const uint32_t a = off[v], b = off[v + 1];
        for (uint32_t e = a + lane; e < b; e += 32) {
            const uint64_t bit = 8ull * a + filter_bit(adj[e] >> lbits, b - a);
            atomicOr(&filter[bit >> 5], 1u << (bit & 31));
        }
    }
}

// Degree moments of one label's vertices, one block per chunk [first, last) of
// its range: out[16 c + 4 a + b] = sum of dout^a din^b (a, b in 0..3), added up in
// a fixed order (the host adds the chunks), so that plans do not vary.
struct MomentChunk {
    uint32_t first, last;
};
constexpr int MOMENT_THREADS = 128;
constexpr uint32_t MOMENT_CHUNK = 4096;
__global__ void __launch_bounds__(MOMENT_THREADS) k_moments(const MomentChunk* chunks, const uint32_t* out_off,
                                                            const uint32_t* in_off, double* out) {
    const MomentChunk c = chunks[blockIdx.x];
    double M[16] = {};
    for (uint32_t v = c.first + threadIdx.x; v < c.last; v += MOMENT_THREADS) {
        const double dout = (double)(out_off[v + 1] - out_off[v]), din = (double)(in_off[v + 1] - in_off[v]);
        double pa = 1.0;
#pragma unroll
        for (int a = 0; a < 4; a++) {
            double pb = pa;
#pragma unroll
            for (int b = 0; b < 4; b++) {
                M[4 * a + b] += pb;
                pb *= din;
            }
            pa *= dout;
        }
    }
    __shared__ double part[MOMENT_THREADS / 32][16];
#pragma unroll
    for (int i = 0; i < 16; i++) {
        double x = M[i];
        for (int d = 16; d >= 1; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5][i] = x;
    }
    __syncthreads();
    if (threadIdx.x < 16) {
        double x = 0;
        for (int w = 0; w < MOMENT_THREADS / 32; w++) x += part[w][threadIdx.x];
        out[16 * (uint64_t)blockIdx.x + threadIdx.x] = x;
    }
}

// One device allocation cut into aligned parts (two per graph: what stays
// resident, and the scratch of the load).
struct Block {
    size_t size = 0;
    uint8_t* base = nullptr;
    size_t take(size_t bytes) {
        const size_t at = size;
        size = (size + std::max<size_t>(bytes, 1) + 255) & ~(size_t)255;
        return at;
    }
    int alloc() {
        const cudaError_t e = cudaMalloc((void**)&base, size);
        if (e != cudaSuccess) {
            cudaGetLastError();
            base = nullptr;
            set_error(GFD_ERR_OUT_OF_MEMORY, "cudaMalloc of %zu bytes failed: %s", size, cudaGetErrorString(e));
            return GFD_ERR_OUT_OF_MEMORY;
        }
        return GFD_OK;
    }
    template <typename T>
    T* at(size_t off) const {
        return reinterpret_cast<T*>(base + off);
    }
};

// written by the load's kernels, read back at its synchronisations
struct Flags {
    uint32_t bad;
    int32_t maxlab;
    uint32_t nsegs;
    uint32_t class_end[N_CLASS - 1];
};

struct TmpFree {
    void* p = nullptr;
    ~TmpFree() {
        if (p) cudaFree(p);
    }
};

// Attribute columns are reordered through scratch of up to this many bytes (one column
// at least): a second copy of them all would keep graphs with many attributes out.
constexpr size_t ATTR_SCRATCH = (size_t)256 << 20;

int grid_for(int64_t n, int threads = 256) {
    int64_t b = (n + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)device_sms() * 16));
}

std::string bad_text(uint32_t bad) {
    std::string s;
    if (bad & BAD_OFFSETS) s += " offsets not a valid CSR;";
    if (bad & BAD_ORDER) s += " adjacency row not strictly increasing (repeated or unsorted edge);";
    if (bad & BAD_RANGE) s += " vertex id out of range;";
    if (bad & BAD_LABEL) s += " label out of range;";
    if (bad & BAD_REVERSE) s += " reverse CSR differs from the transpose of the forward CSR;";
    return s;
}

}  // namespace

int device_sms() {
    static std::mutex mu;
    static std::map<int, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    const auto it = cache.find(dev);
    if (it != cache.end()) return it->second;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        return 1;  // not cached: a later call may succeed
    }
    cache.emplace(dev, sms);
    return sms;
}

int graph_load(const gfd_graph_desc* d, const gfd_opts* o, gfd_graph** out) {
    if (!d || !out) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_graph_load: NULL argument");
        return GFD_ERR_INVALID_ARG;
    }
    const int32_t n = d->n_vertices;
    const int64_t m = d->n_edges;
    if (n < 0 || m < 0 || d->n_attrs < 0 || !d->out_off || (m > 0 && (!d->out_dst || !d->out_elabel)) ||
        (n > 0 && !d->vlabel) || (d->n_attrs > 0 && n > 0 && !d->attrs)) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_graph_load: negative size or missing array");
        return GFD_ERR_INVALID_ARG;
    }
    const bool have_in = d->in_off || d->in_src || d->in_elabel;
    if (have_in && (!d->in_off || (m > 0 && (!d->in_src || !d->in_elabel)))) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_graph_load: reverse CSR given only in part");
        return GFD_ERR_INVALID_ARG;
    }
    if (m >= (int64_t)UINT32_MAX) {
        set_error(GFD_ERR_UNSUPPORTED, "gfd_graph_load: %lld edges, limit is 2^32-1", (long long)m);
        return GFD_ERR_UNSUPPORTED;
    }
    int32_t nb = 1;  // bits of a vertex id
    while ((1ll << nb) < (int64_t)n) nb++;

    cudaStream_t st = o && o->cuda_stream ? (cudaStream_t)o->cuda_stream : nullptr;
    gfd_graph* g = new gfd_graph();
    g->n = n;
    g->m = m;
    g->n_attrs = d->n_attrs;
    auto fail = [&](int code) {
        graph_free(g);
        return code;
    };
    cudaError_t ce = cudaStreamCreateWithFlags(&g->stream, cudaStreamNonBlocking);
    if (ce != cudaSuccess) return fail(cuda_fail(ce, "cudaStreamCreate"));
    if (!st) st = g->stream;

    const size_t N = (size_t)n, M = (size_t)m, NA = N * std::max(1, d->n_attrs);
    Block R;  // resident
    const size_t r_out_off = R.take(4 * (N + 1)), r_in_off = R.take(4 * (N + 1)), r_out_adj = R.take(4 * M + 16),
                 r_in_adj = R.take(4 * M + 16), r_vinfo = R.take(4 * N), r_attrs = R.take(4 * NA), r_sig = R.take(16 * N), r_filter = R.take(2 * (M + 256)),
                 r_orig = R.take(4 * N), r_ovinfo = R.take(4 * N), r_oout = R.take(4 * (N + 1)),
                 r_oin = R.take(4 * (N + 1));
    int rc;
    if ((rc = R.alloc())) return fail(rc);
    g->allocs = {R.base};
    g->bytes = (int64_t)R.size;

    // scratch; the sorts' temporary storage is queried first
    size_t sort_v = 0, sort_e = 0, scan_b = 0;
    {
        cub::DoubleBuffer<uint64_t> kb(nullptr, nullptr);
        cub::DoubleBuffer<uint32_t> vb(nullptr, nullptr);
        cub::DoubleBuffer<uint8_t> lb(nullptr, nullptr);
        cudaError_t e = cub::DeviceRadixSort::SortPairs(nullptr, sort_v, kb, vb, (int64_t)n, 0, KEY_BITS, st);
        if (e == cudaSuccess) e = cub::DeviceRadixSort::SortPairs(nullptr, sort_e, kb, lb, (int64_t)m, 0, 2 * nb, st);
        if (e == cudaSuccess) e = cub::DeviceScan::ExclusiveSum(nullptr, scan_b, (uint32_t*)nullptr, (uint32_t*)nullptr, n + 1, st);
        if (e != cudaSuccess) return fail(cuda_fail(e, "sort scratch size"));
    }
    const size_t cub_bytes = std::max(sort_v, std::max(sort_e, scan_b));
    constexpr size_t LABELS = 65536;
    const int32_t cols = std::min<int32_t>(d->n_attrs, (int32_t)std::max<size_t>(1, ATTR_SCRATCH / (4 * N + 1)));
    Block S;
    const size_t s_off = S.take(8 * (N + 1)), s_nbr = S.take(4 * M), s_lab = S.take(4 * M), s_vl = S.take(4 * N),
                 s_at = S.take(4 * N * cols), s_k0 = S.take(8 * std::max(M, N)), s_k1 = S.take(8 * std::max(M, N)),
                 s_l0 = S.take(std::max(M, 4 * N)), s_l1 = S.take(std::max(M, 4 * N)), s_rank = S.take(4 * N),
                 s_dout = S.take(4 * (N + 1)), s_din = S.take(4 * (N + 1)), s_zero = S.size,
                 s_odin = S.take(4 * (N + 1)), s_self = S.take(4 * N), s_hist = S.take(8 * 256), s_flag = S.take(sizeof(Flags)),
                 s_zend = S.size, s_cub = S.take(cub_bytes);
    // segments, and chunks of the moments: whole ones, and one begun per segment
    const size_t max_segs = std::min(N, N_CLASS * LABELS) + 1, max_chunks = N / MOMENT_CHUNK + max_segs;
    const size_t s_seg = S.take(sizeof(Segment) * max_segs);
    const size_t s_chunk = S.take(sizeof(MomentChunk) * max_chunks), s_mom = S.take(16 * sizeof(double) * max_chunks);
    if ((rc = S.alloc())) return fail(rc);
    TmpFree tmp{S.base};
    int64_t* d_off = S.at<int64_t>(s_off);
    int32_t *d_nbr = S.at<int32_t>(s_nbr), *d_lab = S.at<int32_t>(s_lab), *d_vl = S.at<int32_t>(s_vl);
    Flags* d_flag = S.at<Flags>(s_flag);
    uint32_t *d_bad = &d_flag->bad, *odin = S.at<uint32_t>(s_odin), *self = S.at<uint32_t>(s_self);
    uint32_t *out_off = R.at<uint32_t>(r_out_off), *in_off = R.at<uint32_t>(r_in_off),
             *out_adj = R.at<uint32_t>(r_out_adj), *in_adj = R.at<uint32_t>(r_in_adj),
             *vinfo = R.at<uint32_t>(r_vinfo), *orig = R.at<uint32_t>(r_orig), *o_vinfo = R.at<uint32_t>(r_ovinfo),
             *o_out = R.at<uint32_t>(r_oout), *o_in = R.at<uint32_t>(r_oin);
    int32_t* attrs = R.at<int32_t>(r_attrs);
    unsigned long long* sig = R.at<unsigned long long>(r_sig);
#define CK(call)                                         \
    do {                                                 \
        cudaError_t _e = (call);                         \
        if (_e != cudaSuccess) return fail(cuda_fail(_e, #call)); \
    } while (0)
    CK(cudaMemsetAsync(S.base + s_zero, 0, s_zend - s_zero, st));
    CK(cudaMemcpyAsync(d_off, d->out_off, sizeof(int64_t) * (N + 1), cudaMemcpyHostToDevice, st));
    if (m) {
        CK(cudaMemcpyAsync(d_lab, d->out_elabel, sizeof(int32_t) * M, cudaMemcpyHostToDevice, st));
        k_edge_labels<<<grid_for(m), 256, 0, st>>>(d_lab, m, &d_flag->maxlab, S.at<unsigned long long>(s_hist));
    }
    k_check_offsets<<<grid_for(n + 1), 256, 0, st>>>(d_off, n, m, d_bad);
    Flags flag{};
    unsigned long long hist[256];
    CK(cudaMemcpyAsync(&flag, d_bad, sizeof(flag), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(hist, S.at<void>(s_hist), sizeof(hist), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    // edge-label bit width from the largest label (rows are checked below)
    if (flag.maxlab > 255) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_graph_load: edge label %d > 255", flag.maxlab);
        return fail(GFD_ERR_INVALID_ARG);
    }
    int32_t lbits = 1;
    while ((1 << lbits) <= flag.maxlab) lbits++;
    g->lbits = lbits;
    if ((int64_t)n > (1ll << (32 - lbits))) {
        set_error(GFD_ERR_UNSUPPORTED, "gfd_graph_load: %d vertices with %d-bit edge labels exceed 2^%d",
                  n, lbits, 32 - lbits);
        return fail(GFD_ERR_UNSUPPORTED);
    }
    const uint32_t lmask = (1u << lbits) - 1;
    auto bad_rows = [&](const char* what) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_graph_load:%s%s", what, bad_text(flag.bad).c_str());
        return fail(GFD_ERR_INVALID_ARG);
    };
    if (flag.bad) return bad_rows(" forward CSR:");
    if (m) CK(cudaMemcpyAsync(d_nbr, d->out_dst, sizeof(int32_t) * M, cudaMemcpyHostToDevice, st));
    if (n) CK(cudaMemcpyAsync(d_vl, d->vlabel, sizeof(int32_t) * N, cudaMemcpyHostToDevice, st));
    auto copy_attrs = [&](int32_t a) {  // columns [a, a + cols) of those there are
        return cudaMemcpyAsync(S.at<void>(s_at), d->attrs + (size_t)a * N, sizeof(int32_t) * N * std::min(cols, d->n_attrs - a),
                               cudaMemcpyHostToDevice, st);
    };
    if (n && d->n_attrs) CK(copy_attrs(0));
    cub::DoubleBuffer<uint64_t> kb(S.at<uint64_t>(s_k0), S.at<uint64_t>(s_k1));
    cub::DoubleBuffer<uint32_t> vb(S.at<uint32_t>(s_l0), S.at<uint32_t>(s_l1));
    k_check_rows<<<grid_for((int64_t)n * 32), 256, 0, st>>>(d_off, d_nbr, d_lab, n, lbits, odin, self, d_bad);
    k_vertex_keys<<<grid_for(n), 256, 0, st>>>(d_vl, d_off, odin, self, n, o_vinfo, o_out, kb.Current(), vb.Current(),
                                               d_bad);
    CK(cudaGetLastError());
    // the kernels below index arrays by neighbour id: stop here on a bad row
    CK(cudaMemcpyAsync(&flag, d_bad, sizeof(flag), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (flag.bad) return bad_rows(" forward CSR:");

    size_t tb = cub_bytes;
    void* tstore = S.at<void>(s_cub);
    CK(cub::DeviceScan::ExclusiveSum(tstore, tb, odin, o_in, n + 1, st));
    tb = cub_bytes;
    CK(cub::DeviceRadixSort::SortPairs(tstore, tb, kb, vb, (int64_t)n, 0, KEY_BITS, st));
    CK(cudaMemcpyAsync(orig, vb.Current(), 4 * N, cudaMemcpyDeviceToDevice, st));
    uint32_t *rank = S.at<uint32_t>(s_rank), *dout_new = S.at<uint32_t>(s_dout), *din_new = S.at<uint32_t>(s_din);
    CK(cudaMemsetAsync(dout_new + N, 0, 4, st));
    CK(cudaMemsetAsync(din_new + N, 0, 4, st));
    k_renumber<<<grid_for(n), 256, 0, st>>>(orig, kb.Current(), o_vinfo, d_off, odin, n, rank, vinfo, dout_new, din_new,
                                            S.at<Segment>(s_seg), &d_flag->nsegs, d_flag->class_end);
    for (int32_t a = 0; n && a < d->n_attrs; a += cols) {
        if (a) CK(copy_attrs(a));
        k_gather_attrs<<<grid_for(n), 256, 0, st>>>(S.at<int32_t>(s_at), orig, n, std::min(cols, d->n_attrs - a),
                                                    attrs + (size_t)a * N);
    }
    tb = cub_bytes;
    CK(cub::DeviceScan::ExclusiveSum(tstore, tb, dout_new, out_off, n + 1, st));
    tb = cub_bytes;
    CK(cub::DeviceScan::ExclusiveSum(tstore, tb, din_new, in_off, n + 1, st));
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(&flag, d_flag, sizeof(flag), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    std::vector<Segment> segs(flag.nsegs);
    if (!segs.empty())
        CK(cudaMemcpyAsync(segs.data(), S.at<void>(s_seg), sizeof(Segment) * segs.size(), cudaMemcpyDeviceToHost, st));
    // (0 where all classes up to one are empty: the ends never fall)
    for (int c = 0; c < N_CLASS - 1; c++) g->dg.class_end[c] = std::max(flag.class_end[c], c ? g->dg.class_end[c - 1] : 0u);

    // both adjacency arrays: edges sorted by (source, destination) and by
    // (destination, source) in the inside numbering
    const uint8_t* sorted_labs = nullptr;
    auto sort_edges = [&](const uint32_t* by, bool reverse) -> cudaError_t {
        kb = cub::DoubleBuffer<uint64_t>(S.at<uint64_t>(s_k0), S.at<uint64_t>(s_k1));
        cub::DoubleBuffer<uint8_t> lb(S.at<uint8_t>(s_l0), S.at<uint8_t>(s_l1));
        k_edge_keys<<<grid_for((int64_t)n * 32), 256, 0, st>>>(d_off, d_nbr, d_lab, by, n, nb, reverse, kb.Current(),
                                                              lb.Current());
        size_t b = cub_bytes;
        const cudaError_t e = cub::DeviceRadixSort::SortPairs(tstore, b, kb, lb, (int64_t)m, 0, 2 * nb, st);
        sorted_labs = lb.Current();
        return e == cudaSuccess ? cudaGetLastError() : e;
    };
    for (int rev = 0; rev < 2 && m > 0; rev++) {
        CK(sort_edges(rank, rev != 0));
        k_pack_adj<<<grid_for(m), 256, 0, st>>>(kb.Current(), sorted_labs, m, nb, lbits, rev ? in_adj : out_adj);
    }
    k_signature<<<grid_for((int64_t)n * 32), 256, 0, st>>>(out_off, out_adj, n, lbits, 0, sig);
    k_signature<<<grid_for((int64_t)n * 32), 256, 0, st>>>(in_off, in_adj, n, lbits, 1, sig);
    uint8_t *out_filter = R.at<uint8_t>(r_filter), *in_filter = out_filter + ((M + 255) & ~(size_t)255);
    CK(cudaMemsetAsync(out_filter, 0, 2 * (M + 256), st));
    k_row_filter<<<grid_for((int64_t)n * 32), 256, 0, st>>>(out_off, out_adj, n, lbits, (uint32_t*)out_filter);
    k_row_filter<<<grid_for((int64_t)n * 32), 256, 0, st>>>(in_off, in_adj, n, lbits, (uint32_t*)in_filter);
    CK(cudaGetLastError());
    if (have_in) {
        // the caller's reverse CSR must be exactly the transpose
        if (m) CK(sort_edges(nullptr, true));
        CK(cudaMemcpyAsync(d_off, d->in_off, sizeof(int64_t) * (N + 1), cudaMemcpyHostToDevice, st));
        if (m) {
            CK(cudaMemcpyAsync(d_nbr, d->in_src, sizeof(int32_t) * M, cudaMemcpyHostToDevice, st));
            CK(cudaMemcpyAsync(d_lab, d->in_elabel, sizeof(int32_t) * M, cudaMemcpyHostToDevice, st));
        }
        k_check_offsets<<<grid_for(n + 1), 256, 0, st>>>(d_off, n, m, d_bad);
        CK(cudaMemcpyAsync(&flag, d_bad, sizeof(flag), cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        if (flag.bad) return bad_rows("");
        k_check_rows<<<grid_for((int64_t)n * 32), 256, 0, st>>>(d_off, d_nbr, d_lab, n, lbits, nullptr, nullptr, d_bad);
        k_compare_reverse<<<grid_for((int64_t)n * 32), 256, 0, st>>>(d_off, d_nbr, d_lab, n, nb, o_in, kb.Current(),
                                                                    sorted_labs, d_bad);
        CK(cudaGetLastError());
    }
    // statistics per label: how many vertices, degree sums and moments (the
    // segments were copied before the sorts)
    std::vector<MomentChunk> chunks;
    std::vector<uint32_t> chunk_label;
    uint32_t n_labels = 0;
    CK(cudaStreamSynchronize(st));
    std::sort(segs.begin(), segs.end(), [](const Segment& x, const Segment& y) { return x.first < y.first; });
    for (size_t i = 0; i < segs.size(); i++) {
        const uint32_t last = i + 1 < segs.size() ? segs[i + 1].first : (uint32_t)n;
        n_labels = std::max(n_labels, segs[i].label + 1);
        for (uint32_t v = segs[i].first; v < last; v += std::min(MOMENT_CHUNK, last - v)) {
            chunks.push_back({v, v + std::min(MOMENT_CHUNK, last - v)});
            chunk_label.push_back(segs[i].label);
        }
    }
    g->label_range.assign(n_labels, {});
    for (size_t i = 0; i < segs.size(); i++) {
        int c = 0;
        while (c < N_CLASS - 1 && segs[i].first >= g->dg.class_end[c]) c++;
        g->label_range[segs[i].label][2 * c] = segs[i].first;
        g->label_range[segs[i].label][2 * c + 1] = i + 1 < segs.size() ? segs[i + 1].first : (uint32_t)n;
    }
    g->moments.assign((size_t)n_labels * 16, 0.0);
    g->moments_all.assign(16, 0.0);
    if (!chunks.empty()) {
        double* d_m = S.at<double>(s_mom);
        MomentChunk* d_c = S.at<MomentChunk>(s_chunk);
        std::vector<double> part(16 * chunks.size());
        CK(cudaMemcpyAsync(d_c, chunks.data(), sizeof(MomentChunk) * chunks.size(), cudaMemcpyHostToDevice, st));
        k_moments<<<(unsigned)chunks.size(), MOMENT_THREADS, 0, st>>>(d_c, out_off, in_off, d_m);
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(part.data(), d_m, sizeof(double) * part.size(), cudaMemcpyDeviceToHost, st));
        CK(cudaMemcpyAsync(&flag, d_bad, sizeof(flag), cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        for (size_t c = 0; c < chunks.size(); c++)
            for (int i = 0; i < 16; i++) g->moments[16 * (size_t)chunk_label[c] + i] += part[16 * c + i];
        for (uint32_t L = 0; L < n_labels; L++)
            for (int i = 0; i < 16; i++) g->moments_all[i] += g->moments[16 * (size_t)L + i];
    } else {
        CK(cudaStreamSynchronize(st));
    }
    if (flag.bad) return bad_rows("");
#undef CK
    // count, out-degree sum and in-degree sum of a label are its moments (0, 0),
    // (1, 0) and (0, 1): whole numbers below 2^53, exact in any order
    g->label_stats.assign((size_t)n_labels * 3, 0);
    for (uint32_t L = 0; L < n_labels; L++) {
        g->label_stats[3 * (size_t)L] = (unsigned long long)g->moments[16 * (size_t)L];
        g->label_stats[3 * (size_t)L + 1] = (unsigned long long)g->moments[16 * (size_t)L + 4];
        g->label_stats[3 * (size_t)L + 2] = (unsigned long long)g->moments[16 * (size_t)L + 1];
    }
    g->elabel_frac.assign(256, 0.0);
    for (int l = 0; l < 256; l++) g->elabel_frac[l] = (double)hist[l] / (double)std::max<int64_t>(1, m);
    DevGraph& dg = g->dg;
    dg.n = n;
    dg.n_attrs = d->n_attrs;
    dg.lbits = lbits;
    dg.lmask = lmask;
    dg.m = m;
    dg.nwords = (uint32_t)(((int64_t)n + 31) / 32);
    dg.out_off = out_off;
    dg.in_off = in_off;
    dg.out_adj = out_adj;
    dg.in_adj = in_adj;
    dg.vinfo = vinfo;
    dg.attrs = attrs;
    dg.sig = (const ulonglong2*)sig;
    dg.out_filter = out_filter;
    dg.in_filter = in_filter;
    dg.orig = orig;
    dg.o_vinfo = o_vinfo;
    dg.o_out_off = o_out;
    dg.o_in_off = o_in;
    *out = g;
    return GFD_OK;
}

void graph_free(gfd_graph* g) {
    if (!g) return;
    if (g->eng) engine_free(g->eng);
    for (void* p : g->allocs) cudaFree(p);
    if (g->stream) cudaStreamDestroy(g->stream);
    cudaGetLastError();  // a failure here must not surface in a later, unrelated call
    delete g;
}

}  // namespace gfd
