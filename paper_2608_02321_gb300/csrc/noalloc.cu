// gfd_node_candidates_noalloc: the candidate filter of one pattern node
// (label, degree and self-loop test), computed without allocating any device
// memory. It is meant for callers that may not allocate: a server whose device
// memory is handed out by its own allocator or reserved up front under a fixed
// budget (a library cudaMalloc would bypass that accounting, or fail once the
// reservation holds the free memory), and latency-bound threads that cannot
// wait for cudaFree, which synchronises the whole device. The caller passes
// the graph handle (already resident), the GFD, and a device buffer for the
// output; the only temporary storage is the file-scope array below.
//
// The kernel is a single-pass, order-preserving stream compaction: blocks take
// tiles of consecutive vertices in order from an atomic counter, count the
// vertices that pass, and chain the tile totals with a decoupled look-back over
// per-tile descriptors. Those descriptors, the tile counter, an error word and
// the total are the scratch memory: NA_MAX_TILES tiles of 8192 vertices, so at
// most 2^26 vertices (64 KiB of descriptors plus 64 bytes of counters). Every
// GPU that loads the library keeps this array until the process exits.
//
// Bound: 12 bytes read per vertex and 4 written per candidate, a stream. A lane
// takes four consecutive vertices per round (one 16-byte load per array, a warp
// covers 128 vertices in whole lines; the neighbour lane's first offset closes
// the last degree), and a whole warp looks back over 32 descriptors at a time:
// with one thread walking them, the blocks of the first wave waited for a chain
// of as many L2 round trips. Measured for the whole call, 16M vertices with 3.0M
// candidates: 288 us with 32 vertices per thread (lanes 128 bytes apart) and the
// serial look-back, 118 us with four blocks per multiprocessor, 100 us with
// eight; 20k vertices (one round per tile, 20 blocks): 63 -> 46 us.
#include <algorithm>
#include <cstdio>
#include <mutex>

#include "engine.h"

namespace gfd {

namespace {

constexpr int NA_THREADS = 256;
constexpr int NA_ROUND = NA_THREADS * 4;          // vertices per round of a block
constexpr int NA_ROUNDS = 8;                      // rounds per tile of a large graph
constexpr int NA_TILE = NA_ROUND * NA_ROUNDS;
constexpr int NA_MAX_TILES = 8192;                // => at most 2^26 vertices
constexpr int NA_HEADER = 8;                      // counter words before the descriptors
constexpr uint64_t NA_FLAG_AGG = 1ull << 62;      // tile total published
constexpr uint64_t NA_FLAG_PREFIX = 1ull << 63;   // inclusive prefix published
constexpr uint64_t NA_VALUE = (1ull << 62) - 1;

// [0] tile counter, [1] error (1 = a look-back wait gave up), [2] total count,
// [NA_HEADER + t] descriptor of tile t. Zeroed by every call before its launch.
static __device__ __align__(256) unsigned long long g_na_scratch[NA_HEADER + NA_MAX_TILES];

std::mutex g_na_mu;
void* g_na_ptr[64] = {};  // device address of g_na_scratch, per device
int g_na_sms[64] = {};    // multiprocessor count, per device

// Sum of the totals of the tiles before t (whole warp): from the nearest tile
// with a published inclusive prefix, 32 descriptors at a time, every lane
// waiting (bounded) for its own.
__device__ uint64_t look_back(volatile unsigned long long* desc, uint32_t t, unsigned long long* err, int lane) {
    uint64_t prefix = 0;
    for (int64_t j = (int64_t)t - 1; j >= 0; j -= 32) {
        const int64_t mine = j - lane;
        uint64_t d = mine < 0 ? NA_FLAG_PREFIX : desc[mine];  // before the first tile: an inclusive prefix of 0
        uint64_t spins = 0;
        while (!(d & (NA_FLAG_PREFIX | NA_FLAG_AGG))) {
            if (++spins > (1ull << 22)) {  // bounded wait: give up, report
                atomicExch(err, 1ull);
                d = NA_FLAG_PREFIX;
                break;
            }
            __nanosleep(20);
            d = desc[mine];
        }
        // totals up to the first inclusive prefix (lane 0 is the nearest tile)
        const uint32_t done = __ballot_sync(0xffffffffu, (d & NA_FLAG_PREFIX) != 0);
        const int last = done ? __ffs(done) - 1 : 31;
        uint64_t x = lane <= last ? (d & NA_VALUE) : 0;
        for (int s = 16; s >= 1; s >>= 1) x += __shfl_xor_sync(0xffffffffu, x, s);
        prefix += x;
        if (done) break;
    }
    return prefix;
}

// ROUNDS rounds of NA_ROUND vertices per tile: 8 (each warp streams 1024
// consecutive vertices), or 1 while the tiles of a small graph are fewer than
// the blocks that can run at once.
template <int ROUNDS>
__global__ void __launch_bounds__(NA_THREADS)
k_node_candidates(DevGraph g, FilterKey key, unsigned long long* scratch, int32_t* out, uint64_t cap,
                  uint32_t ntiles) {
    constexpr int WARPS = NA_THREADS / 32;
    __shared__ uint32_t warp_s[WARPS];
    __shared__ uint32_t tile_s;
    __shared__ uint64_t base_s;
    volatile unsigned long long* desc = scratch + NA_HEADER;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n = (uint32_t)g.n;
    for (;;) {
        if (threadIdx.x == 0) tile_s = (uint32_t)atomicAdd(&scratch[0], 1ull);
        __syncthreads();
        const uint32_t t = tile_s;
        if (t >= ntiles) return;
        // the warp's ROUNDS x 128 consecutive vertices, four per lane and round
        const uint32_t w0 = (t * WARPS + warp) * (ROUNDS * 128);
        uint32_t mask = 0, count = 0;  // mask: bit 4 r + c = the c-th vertex of round r passes
#pragma unroll
        for (int r = 0; r < ROUNDS; r++) {
            const uint32_t v = w0 + r * 128 + lane * 4;
            uint32_t vi[4], oo[5], io[5];
            if (v + 4 <= n) {
                const uint4 a = *reinterpret_cast<const uint4*>(g.o_vinfo + v);
                const uint4 o = *reinterpret_cast<const uint4*>(g.o_out_off + v);
                const uint4 i = *reinterpret_cast<const uint4*>(g.o_in_off + v);
                vi[0] = a.x, vi[1] = a.y, vi[2] = a.z, vi[3] = a.w;
                oo[0] = o.x, oo[1] = o.y, oo[2] = o.z, oo[3] = o.w;
                io[0] = i.x, io[1] = i.y, io[2] = i.z, io[3] = i.w;
            } else {  // the graph's last vertices: offsets have n + 1 entries
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    vi[c] = v + c < n ? g.o_vinfo[v + c] : 0u;
                    oo[c] = v + c <= n ? g.o_out_off[v + c] : 0u;
                    io[c] = v + c <= n ? g.o_in_off[v + c] : 0u;
                }
            }
            oo[4] = __shfl_down_sync(0xffffffffu, oo[0], 1);
            io[4] = __shfl_down_sync(0xffffffffu, io[0], 1);
            if (lane == 31) {
                oo[4] = v + 4 <= n ? g.o_out_off[v + 4] : 0u;
                io[4] = v + 4 <= n ? g.o_in_off[v + 4] : 0u;
            }
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const bool has_self = (vi[c] >> 16) != 0;
                const int32_t self_lab = (int32_t)(vi[c] >> 16) - 1;
                const uint32_t dout = oo[c + 1] - oo[c] - has_self;
                const uint32_t din = io[c + 1] - io[c] - has_self;
                const bool self_ok = key.self_exp == EXP_NONE ? !has_self
                                   : key.self_exp == EXP_ANY  ? has_self
                                                              : (has_self && self_lab == key.self_exp);
                const bool p = v + c < n && label_ok(key.label, (int32_t)(vi[c] & 0xffffu)) &&
                               dout >= key.dout_min && din >= key.din_min && self_ok;
                mask |= (uint32_t)p << (4 * r + c);
            }
        }
        count = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(mask));
        if (lane == 0) warp_s[warp] = count;
        __syncthreads();
        uint32_t before = 0, total = 0;  // candidates of the block's earlier warps, of the tile
#pragma unroll
        for (int w = 0; w < WARPS; w++) {
            before += w < warp ? warp_s[w] : 0u;
            total += warp_s[w];
        }
        if (warp == 0) {
            if (lane == 0) {
                desc[t] = (t == 0 ? NA_FLAG_PREFIX : NA_FLAG_AGG) | total;
                __threadfence();
            }
            __syncwarp();
            const uint64_t prefix = look_back(desc, t, &scratch[1], lane);
            if (lane == 0) {
                if (t > 0) desc[t] = NA_FLAG_PREFIX | (prefix + total);
                if (t == ntiles - 1) scratch[2] = prefix + total;
                base_s = prefix;
            }
        }
        __syncthreads();
        uint64_t o = base_s + before;
#pragma unroll
        for (int r = 0; r < ROUNDS; r++) {
            const uint32_t m = (mask >> (4 * r)) & 15u;
            uint32_t excl = 0, all = 0;  // candidates of the round in the lanes before, in the warp
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const uint32_t b = __ballot_sync(0xffffffffu, (m >> c) & 1u);
                excl += __popc(b & ((1u << lane) - 1u));
                all += __popc(b);
            }
            uint64_t p = o + excl;
            const uint32_t v = w0 + r * 128 + lane * 4;
#pragma unroll
            for (int c = 0; c < 4; c++)
                if ((m >> c) & 1u) {
                    if (p < cap) out[p] = (int32_t)(v + c);
                    p++;
                }
            o += all;
        }
        __syncthreads();  // tile_s, warp_s and base_s are reused
    }
}

// Device address of the scratch array on the current device and the device's
// multiprocessor count, looked up once per device (the host-side symbol is only
// a stand-in for the array and must never be handed to a kernel).
int scratch_ptr(unsigned long long** out, int* sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= 64) {
        set_error(GFD_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
        return GFD_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(g_na_mu);
    if (!g_na_ptr[dev]) {
        int n_sm = 0;
        e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute(multiprocessors)");
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_na_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(scratch)");
        g_na_sms[dev] = n_sm > 0 ? n_sm : 1;
        g_na_ptr[dev] = p;
    }
    *out = (unsigned long long*)g_na_ptr[dev];
    *sms = g_na_sms[dev];
    return GFD_OK;
}

}  // namespace

int node_candidates_noalloc(const gfd_graph* g, const gfd_gfd* phi, int32_t node, int32_t* d_out,
                            int64_t out_cap, int64_t* n_out, void* cuda_stream) {
    if (!g || !phi || !n_out || out_cap < 0 || (out_cap > 0 && !d_out)) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_node_candidates_noalloc: NULL argument or negative capacity");
        return GFD_ERR_INVALID_ARG;
    }
    if (node < 0 || node >= phi->k) {
        set_error(GFD_ERR_INVALID_ARG, "gfd_node_candidates_noalloc: node %d outside the pattern", node);
        return GFD_ERR_INVALID_ARG;
    }
    if (((uint64_t)g->n + NA_TILE - 1) / NA_TILE > (uint64_t)NA_MAX_TILES) {
        set_error(GFD_ERR_UNSUPPORTED,
                  "gfd_node_candidates_noalloc: %d vertices exceed the fixed scratch limit of %llu", g->n,
                  (unsigned long long)NA_MAX_TILES * NA_TILE);
        return GFD_ERR_UNSUPPORTED;
    }
    HostPlan plan;  // host memory only
    if (int rc = make_plan(phi, g->n_attrs, g->plan_stats(), &plan)) return rc;
    const FilterKey key = plan.key[plan.level_of[node]];
    unsigned long long* scratch = nullptr;
    int sms = 1;
    if (int rc = scratch_ptr(&scratch, &sms)) return rc;
    cudaStream_t st = cuda_stream ? (cudaStream_t)cuda_stream : g->stream;
    // eight resident blocks per multiprocessor take the tiles in order; one round
    // per tile while that gives no more tiles than blocks
    const uint64_t resident = (uint64_t)sms * 8;
    const uint64_t rounds_small = ((uint64_t)g->n + NA_ROUND - 1) / NA_ROUND;
    const bool small = rounds_small <= std::min<uint64_t>(resident, NA_MAX_TILES);
    const uint64_t ntiles = small ? rounds_small : ((uint64_t)g->n + NA_TILE - 1) / NA_TILE;
    cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(unsigned long long) * (NA_HEADER + ntiles), st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync(scratch)");
    if (ntiles > 0) {
        const int grid = (int)std::min<uint64_t>(ntiles, resident);
        if (small)
            k_node_candidates<1><<<grid, NA_THREADS, 0, st>>>(g->dg, key, scratch, d_out, (uint64_t)out_cap,
                                                              (uint32_t)ntiles);
        else
            k_node_candidates<NA_ROUNDS><<<grid, NA_THREADS, 0, st>>>(g->dg, key, scratch, d_out, (uint64_t)out_cap,
                                                                      (uint32_t)ntiles);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "k_node_candidates");
    }
    unsigned long long hdr[3] = {0, 0, 0};
    e = cudaMemcpyAsync(hdr, scratch, sizeof(hdr), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "gfd_node_candidates_noalloc readback");
    if (hdr[1]) {
        set_error(GFD_ERR_TIMEOUT, "gfd_node_candidates_noalloc: a look-back wait gave up");
        return GFD_ERR_TIMEOUT;
    }
    *n_out = (int64_t)hdr[2];
    if ((int64_t)hdr[2] > out_cap) {
        set_error(GFD_ERR_OVERFLOW, "gfd_node_candidates_noalloc: %llu candidates, output holds %lld",
                  (unsigned long long)hdr[2], (long long)out_cap);
        return GFD_ERR_OVERFLOW;
    }
    return GFD_OK;
}

}  // namespace gfd

extern "C" int gfd_node_candidates_noalloc(const gfd_graph* g, const gfd_gfd* phi, int32_t node, int32_t* d_out,
                                           int64_t out_cap, int64_t* n_out, void* cuda_stream) {
    return gfd::node_candidates_noalloc(g, phi, node, d_out, out_cap, n_out, cuda_stream);
}
