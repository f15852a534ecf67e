// search.cu -- batched K-NN-SEARCH (arXiv:1603.09320, Alg. 5) on one GPU.
//
// One warp answers one query at a time; warps pull query indexes from a
// device work counter until the batch is exhausted (persistent kernel).  Small
// batches take a block of warps per query (search_team.cuh; team_warps below).
//
// Per query:
//   1. greedy ef=1 descent through layers L..1 (Alg. 5's descent).  Under key
//      order (distance, id), SEARCH-LAYER with ef=1 is steepest descent: move
//      to the best of the current element's neighbours while it beats the
//      current element.  No visited set is needed for that.
//   2. SEARCH-LAYER(q, ep, ef', 0) (Alg. 2, ef' = max(ef, K)) as ONE list W in
//      shared memory, sorted by key and capped at ef', with an "expanded" bit
//      per entry instead of the two priority queues: under key order the
//      unextracted candidates that can still be expanded before Alg. 2's
//      stop test fires are exactly the unexpanded entries of W, so "extract
//      the nearest of C" is "take the first unexpanded entry" and the loop
//      ends when none is left.  All unvisited neighbours of the expanded
//      element are scored together and merged at once; inserting them one at
//      a time by Alg. 2's admission and eviction leaves the same top-ef' of
//      the union.
//   3. the K first entries of W (Alg. 5's result), or, with rerank, the K best
//      of W by exact fp32 distance recomputed from the fp32 copy.
//
// Visited set: a 4-way bucketed hash of element ids in shared memory; when a
// bucket is full one of its slots is overwritten, and two lanes storing into
// the same free slot at the same instant keep only one id, so the set may
// FORGET an element.  (The block-per-query kernel tries eight buckets before it
// overwrites, and stores again what it lost to another lane: search_team.cuh,
// visit_all.)  Forgetting never changes the result: an element met again is
// either already in W (its key equals an entry's key and the merge drops it)
// or, being outside W after it was visited, has a key above the furthest entry
// of a full W and is rejected.
// It only costs a repeated distance evaluation, counted in n_eval.
//
// Distances: each row is read as 16-byte chunks by a team of TEAM lanes
// (consecutive lanes read consecutive chunks, so a team's load of one row is
// one contiguous segment), U rows per team in flight, partial sums reduced by
// warp shuffles inside the team.  fp32 accumulation throughout.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <utility>

#include "common.hpp"
#include "index.cuh"
#include "search_kernel.cuh"
#include "search_team.cuh"
#include "stopnet.cuh"

namespace hnswgb {

constexpr int kMaxDeg = 64;  // neighbour slots scored per expansion
static_assert(kMaxDeg == kMaxNbr, "the per-warp layout holds kMaxNbr slots");

// ---- ordering of the second pass --------------------------------------------
// Queries whose upper-layer descent ends far from them tend to need more
// layer-0 expansions; starting them first shortens the tail of the batch
// (longest-first list scheduling).  The order need not be exact: one block
// takes a chunk of up to kSortChunk queries and places them by a counting
// sort into kOrderBuckets buckets spanning the chunk's range of descent
// distances (linear in the distances' ordered bit patterns, so about
// logarithmic in the distances), farthest first; chunks are ordered
// independently.  Block barriers only (no spin-waits); launched with one
// thread per bucket.
constexpr int kSortChunk = 16384;
constexpr int kOrderBuckets = 1024;
static_assert(kOrderBuckets == 1024, "the prefix sum takes one bucket per thread of a 1024-thread block");

__global__ void __launch_bounds__(1024) order_by_descent(const uint64_t* __restrict__ ep_keys, uint32_t n,
                                                        uint32_t* __restrict__ order) {
    __shared__ uint32_t hist[kOrderBuckets];
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t range[2];
    const uint32_t base = blockIdx.x * uint32_t(kSortChunk);
    const uint32_t m = min(uint32_t(kSortChunk), n - base);
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    for (int i = t; i < kOrderBuckets; i += blockDim.x) hist[i] = 0u;
    if (t == 0) {
        range[0] = ~0u;
        range[1] = 0u;
    }
    __syncthreads();
    // the chunk's range of ordered distance bits (the high word of a key)
    uint32_t lo = ~0u, hi = 0u;
    for (uint32_t i = t; i < m; i += blockDim.x) {
        const uint32_t v = uint32_t(ep_keys[base + i] >> 32);
        lo = min(lo, v);
        hi = max(hi, v);
    }
    lo = __reduce_min_sync(kFull, lo);
    hi = __reduce_max_sync(kFull, hi);
    if (lane == 0) {
        atomicMin(&range[0], lo);
        atomicMax(&range[1], hi);
    }
    __syncthreads();
    lo = range[0];
    hi = range[1];
    const uint64_t span = uint64_t(hi - lo) + 1u;  // >= 1 (m >= 1)
    // bucket of a key: 0 for the farthest enter point
    auto bucket = [&](uint32_t i) {
        const uint32_t v = uint32_t(ep_keys[base + i] >> 32);
        return uint32_t((uint64_t(hi - v) * uint64_t(kOrderBuckets)) / span);
    };
    for (uint32_t i = t; i < m; i += blockDim.x) atomicAdd(&hist[bucket(i)], 1u);
    __syncthreads();
    // exclusive prefix sum of the histogram (one entry per thread)
    const uint32_t x = t < kOrderBuckets ? hist[t] : 0u;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        const int nw = int(blockDim.x) >> 5;
        uint32_t w = lane < nw ? wsum[lane] : 0u, wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < nw) wsum[lane] = wi - w;  // exclusive over warps
    }
    __syncthreads();
    if (t < kOrderBuckets) hist[t] = wsum[wid] + inc - x;
    __syncthreads();
    // scatter: the slots of a bucket go to its queries in any order
    for (uint32_t i = t; i < m; i += blockDim.x) order[base + atomicAdd(&hist[bucket(i)], 1u)] = base + i;
}

// ---- host side --------------------------------------------------------------
namespace {

bool is_device_ptr(const void* p) {
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

int ceil_log2(uint64_t x) {
    int r = 0;
    while ((1ull << r) < x) ++r;
    return r;
}

int current_device() {
    int dev = 0;
    cudaGetDevice(&dev);
    return dev;
}

// Blocks of `threads` threads and `smem` bytes of kernel fn resident per SM
// (negative: the query failed).  Cached per (device, kernel, threads, size).
int blocks_per_sm(KernelFn fn, int threads, size_t smem) {
    static std::mutex mu;
    static std::map<std::tuple<int, const void*, int, size_t>, int> cache;
    const auto key = std::make_tuple(current_device(), reinterpret_cast<const void*>(fn), threads, smem);
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    cache[key] = b;
    return b;
}

int sm_count() {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, current_device());
    return sms;
}

// Warps per block (1..8) that put the most warps of kernel fn on an SM
// given `warp_smem` bytes of shared memory per warp (the fewest warps per
// block among equals: finer-grained blocks), and the blocks per SM then.
// Small per-warp state is bound by registers (4-warp blocks); a wide beam's
// state is bound by shared memory, where the block size decides how much of
// an SM's 228 KB the blocks fill.  Cached per (device, kernel, size): a launch
// with an automatic visited set asks for up to six sizes (without this, eight
// look-ups for each: 1 to 4 us of a call).
bool block_choice(KernelFn fn, size_t warp_smem, int& warps, int& per_sm) {
    static std::mutex mu;
    static std::map<std::tuple<int, const void*, size_t>, std::pair<int, int>> cache;
    const auto key = std::make_tuple(current_device(), reinterpret_cast<const void*>(fn), warp_smem);
    {
        std::lock_guard<std::mutex> lk(mu);
        const auto it = cache.find(key);
        if (it != cache.end()) {
            warps = it->second.first;
            per_sm = it->second.second;
            return true;
        }
    }
    int best = 0;
    warps = 0;
    per_sm = 0;
    for (int w : {4, 5, 6, 7, 8, 3, 2, 1}) {
        const size_t sm = size_t(w) * warp_smem;
        if (sm > 227 * 1024) continue;
        const int b = blocks_per_sm(fn, w * 32, sm);
        if (b < 0) return false;
        if (b * w > best) {
            best = b * w;
            warps = w;
            per_sm = b;
        }
    }
    if (best == 0) return false;
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = {warps, per_sm};
    return true;
}

// The instantiation for an index's stored rows (null: none).
KernelFn search_kernel(const DevIndex& D, KernelAsk k) {
    k.chunks = D.row_chunks;
    switch (D.storage) {
        case HNSW_F32: return search_kernel_f32(k);
        case HNSW_BF16: return search_kernel_bf16(k);
        case HNSW_F16: return search_kernel_f16(k);
        case HNSW_FP8E4M3: return search_kernel_fp8(k);
    }
    return nullptr;
}

}  // namespace

// Upper bound of the automatic visited set: about 8-16 slots per beam entry,
// 1,024 to 4,096 slots (a layer-0 search evaluates some 10-30 x ef'
// elements); the launch takes the largest size up to it that costs no
// resident warps, and not below kMinAutoHlog.
constexpr int kMinAutoHlog = 8;
int auto_visited_log2(int efp) {
    int l = ceil_log2(uint64_t(efp) * 8);
    return l < 10 ? 10 : (l > 12 ? 12 : l);
}

// The scheduling scratch (two passes, deferral) comes from the device's
// default stream-ordered pool, which by default hands freed memory back at
// every synchronisation, so that the next call maps it again.  This process
// keeps up to 256 MB of it cached (an attribute of the process's pool,
// nothing of the device's settings).
#ifndef HNSW_POOL_KEEP
#define HNSW_POOL_KEEP 1
#endif
void keep_pool_memory() {
#if HNSW_POOL_KEEP
    static std::mutex mu;
    static std::map<int, bool> done;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    std::lock_guard<std::mutex> g(mu);
    if (done[dev]) return;
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
        uint64_t thr = 256ull << 20;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    cudaGetLastError();
    done[dev] = true;
#endif
}

// Deferral of a launch: none, when some warp takes several queries, always.
enum class Defer { no, automatic, always };

// Warps per query of the block-per-query kernel for this search, or 0: a warp
// per query.  The block kernel shortens a query's chain but spends more
// instructions and registers on it, so it is taken while all queries of the
// batch are resident at once: up to two 8-warp blocks per SM, then up to four
// 4-warp blocks (both sides of the limits: search_team.cuh).  Beams above 256
// keep more of W in registers and shared memory: three 4-warp blocks (ef 498,
// warp per query / block: 400 queries 1.24 times the time, 608 on GloVe-shaped
// data 0.83 to 0.88 times).  Rows of up to 32 bytes leave little to score
// ahead: without rerank a warp per query is as quick or quicker above ef 64 (8
// fp32 coordinates, ef 200, 8 queries: block 298 us, warp 266), with rerank
// above ef 256 (8 f16 coordinates, block / warp: ef 257, 40 queries 559 / 464,
// 400 queries 842 / 755; ef 498, 400 queries 1,300 / 1,246; but ef 256, 77
// queries 448 / 513).
int team_warps(const DevIndex& D, const hnsw_search_params& p, uint32_t n) {
    const int efp = std::max(p.ef, p.k);
    if (p.schedule != 0 || p.check_bounds || D.N == 0 || D.N >= kTeamMaxN || efp > 512) return 0;
    if (D.row_chunks <= 2 && efp > (p.rerank ? 256 : 64)) return 0;
    const uint32_t sms = uint32_t(sm_count());
    return n <= 2 * sms ? 8 : n <= (efp > 256 ? 3 : 4) * sms ? 4 : 0;
}

// Launches the block-per-query kernel fn with nw warps per block on the
// arguments filled in so far.
hnsw_status launch_team(SearchArgs& a, KernelFn fn, int nw, int visited_log2, cudaStream_t s) {
    const uint32_t slots = (std::max(a.ix.Mmax0, a.ix.Mmax) + 31u) & ~31u;
    const size_t row32 = size_t(a.ix.row_chunks32) * 16;
    auto layout = [&](int hl) {
        // the visited set; after the search its bytes hold W and, for the
        // rerank, a copy of q
        a.hlog = hl;
        a.off_vis = 0;
        a.off_qs = a.efcap * 8;
        size_t o = std::max(size_t(4) << hl, size_t(a.efcap) * 8 + (a.rerank ? row32 : 0));
        a.off_slot = int(o);
        o += size_t(nw) * 2 * slots * 4;
        a.off_merge = int(o);
        o += size_t(32 + (a.efcap <= 64 ? 64 : a.efcap <= 256 ? 256 : 512)) * 8;
        a.off_ctl = int(o);
        o += (sizeof(TeamCtl) + 15) & ~size_t(15);
        return o;
    };
    const int sms = sm_count();
    auto resident = [&](size_t smem) { return uint64_t(std::max(0, blocks_per_sm(fn, nw * 32, smem))) * sms; };
    const int most = visited_log2 > 0 ? visited_log2 : std::min(14, std::max(11, ceil_log2(uint64_t(a.efp) * 64)));
    if (layout(most) > 227 * 1024) return fail(HNSW_EINVAL, "search: ef/visited set too large for shared memory");
    const hnsw_status st = raise_smem_limit(reinterpret_cast<const void*>(fn), layout(most), "search");
    if (st != HNSW_OK) return st;
    int hl = most;
    if (visited_log2 <= 0) {
        // the largest set that keeps as many queries resident as the smallest
        // one does, or all of them
        const uint64_t want = std::min<uint64_t>(a.n, resident(layout(10)));
        while (hl > 10 && resident(layout(hl)) < want) --hl;
    }
    const size_t smem = layout(hl);
    const uint64_t cap = resident(smem);
    if (cap == 0) return fail(HNSW_ECUDA, "search: occupancy query failed");
    const unsigned grid = unsigned(std::min<uint64_t>(a.n, cap));
    cudaError_t e = cudaSuccess;
    if (a.n > grid) e = cudaMemsetAsync(a.work, 0, 4, s);
    if (e == cudaSuccess) {
        fn<<<grid, nw * 32, smem, s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return fail(HNSW_ECUDA, std::string("search launch: ") + cudaGetErrorString(e));
    return HNSW_OK;
}

hnsw_status launch_search_mode(hnsw_index* ix, const hnsw_search_params& p, const float* q, uint32_t n,
                               uint32_t* ids, float* dists, hnsw_query_stats* stats, cudaStream_t s,
                               uint32_t* work, const StopModel* stop, int mode, uint64_t* ep_keys,
                               uint32_t* up_cnt, const uint32_t* order, const uint32_t* q_kef = nullptr,
                               const uint64_t* q_out = nullptr, const DevIndex* view = nullptr,
                               Defer defer = Defer::no) {
    const DevIndex D = view ? *view : dev_snapshot(ix);
    if (p.check_bounds && stop != nullptr)
        return fail(HNSW_EINVAL, "search: check_bounds with the learned stop or a trace");
    SearchArgs a{};
    a.ix = D;
    a.q = q;
    a.n = n;
    a.k = p.k;
    a.efp = p.ef > p.k ? p.ef : p.k;
    a.efcap = 1 << ceil_log2(uint64_t(a.efp < 32 ? 32 : a.efp));
    const bool stop_build = stop != nullptr && stop->period > 0;
    const int team = mode == 0 && !stop && defer != Defer::always ? team_warps(D, p, n) : 0;
    const KernelFn fn = search_kernel(D, {0, stop_build, a.efcap > 64 || D.Mmax0 > 32, p.check_bounds != 0,
                                        team ? (a.efcap <= 64 ? 2 : a.efcap <= 256 ? 8 : 16) : 0});
    if (!fn)
        return fail(HNSW_EINVAL, p.check_bounds ? "search: check_bounds is built for f32 rows of d <= 128 and bf16 of d <= 128"
                                                : "search: unsupported row size");
    a.rerank = p.rerank;
    a.out_ids = ids;
    a.out_dists = dists;
    a.stats = stats;
    a.work = work;
    a.mode = mode;
    a.q_kef = q_kef;
    a.q_out = q_out;
    a.ep_keys = ep_keys;
    a.up_cnt = up_cnt;
    a.order = order;
    a.dfr_hold = ix->hold_decisions.load() ? 1 : 0;
    a.err = ix->d_err;
    if (stop) {
        a.stop = static_cast<const StopDev*>(stop->stop);
        a.stop_logit = stop->logit_threshold;
        a.stop_period = stop->period;
        a.tr_feat = stop->tr_feat;
        a.tr_topk = stop->tr_topk;
        a.tr_logit = stop->tr_logit;
        a.tr_count = stop->tr_count;
        a.tr_max = stop->tr_max;
    }
    if (team) return launch_team(a, fn, team, p.visited_log2, s);
    const size_t row32 = size_t(D.row_chunks32) * 16;
    // per-warp layout with a visited set of 2^hl slots (every piece a
    // multiple of 16 bytes); sets the offsets in t, returns the bytes
    auto layout = [&](int hl, SearchArgs& t) {
        const size_t hbytes = (size_t(1) << hl) * 4;
        size_t per_warp = size_t(t.efcap) * 8 + hbytes + kMaxDeg * 12 + 64;
        t.off_hs = int(per_warp);
        if (stop_build) per_warp += size_t(kStopH) * 4;
        if (!p.rerank || hbytes >= row32) {
            t.off_qs = t.efcap * 8;  // the visited set's bytes
        } else {
            t.off_qs = int(per_warp);
            per_warp += row32;
        }
        return per_warp;
    };
    int hl = p.visited_log2 > 0 ? p.visited_log2 : auto_visited_log2(a.efp);
    if (p.visited_log2 <= 0) {
        // automatic: the largest set, down to 2^8 slots, that keeps as many
        // warps resident as the smallest does.  A forgotten element only
        // costs a repeated evaluation, while the warps resident decide how
        // much of the gathers' latency is hidden (a wide beam's state is
        // bound by shared memory, a narrow one's by registers).
        SearchArgs t = a;
        const size_t most = std::min<size_t>(227 * 1024, size_t(8) * layout(hl, t));
        const hnsw_status st = raise_smem_limit(reinterpret_cast<const void*>(fn), most, "search");
        if (st != HNSW_OK) return st;
        int w0 = 0, b0 = 0;
        if (!block_choice(fn, layout(kMinAutoHlog, t), w0, b0))
            return fail(HNSW_ECUDA, "search: occupancy query failed");
        for (; hl > kMinAutoHlog; --hl) {
            const size_t pw = layout(hl, t);
            int w = 0, b = 0;
            if (pw <= 227 * 1024 && block_choice(fn, pw, w, b) && w * b >= w0 * b0) break;
        }
    }
    a.hlog = hl;
    const size_t per_warp = layout(hl, a);
    a.warp_smem = int(per_warp);
    if (size_t(a.warp_smem) > 227 * 1024)
        return fail(HNSW_EINVAL, "search: ef/visited set too large for shared memory");
    const int sms = sm_count();
    int per_sm = 0, warps = 0;
    {
        const size_t most = std::min<size_t>(227 * 1024, size_t(8) * a.warp_smem);
        const hnsw_status st = raise_smem_limit(reinterpret_cast<const void*>(fn), most, "search");
        if (st != HNSW_OK) return st;
    }
    if (!block_choice(fn, size_t(a.warp_smem), warps, per_sm))
        return fail(HNSW_ECUDA, "search: occupancy query failed");
    const size_t smem = size_t(warps) * a.warp_smem;
    const uint64_t need = (uint64_t(n) + warps - 1) / warps;
    const uint64_t cap = uint64_t(per_sm) * uint64_t(sms);
    const unsigned grid = unsigned(need < cap ? need : cap);
    // deferral orders the work of warps that take several queries: with a
    // warp for every query it only adds waits (measured at 77 queries, bf16
    // rows: 466 us against 308)
    const bool dfr = defer == Defer::always || (defer == Defer::automatic && need > cap);
    cudaError_t e = cudaSuccess;
    void* scr = nullptr;
    if (dfr) {
        // stream-ordered scratch: control words (64 bytes, zero) and one
        // 16-byte record per query (all ones until written)
        const size_t bc = 256, br = al256(size_t(n) * 16);
        keep_pool_memory();
        if (cudaMallocAsync(&scr, bc + br, s) != cudaSuccess) {
            cudaGetLastError();
            return fail(HNSW_ENOMEM, "hnsw_search: scheduling scratch");
        }
        a.dfr_ctl = static_cast<uint32_t*>(scr);
        a.dfr_rec = reinterpret_cast<uint4*>(static_cast<char*>(scr) + bc);
        e = cudaMemsetAsync(a.dfr_ctl, 0, bc, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(a.dfr_rec, 0xff, br, s);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(work, 0, 4, s);
    if (e == cudaSuccess) {
        fn<<<grid, warps * 32, smem, s>>>(a);
        e = cudaGetLastError();
    }
    if (scr) cudaFreeAsync(scr, s);
    if (e != cudaSuccess) return fail(HNSW_ECUDA, std::string("search launch: ") + cudaGetErrorString(e));
    return HNSW_OK;
}

hnsw_status launch_search(hnsw_index* ix, const hnsw_search_params& p, const float* q, uint32_t n,
                          uint32_t* ids, float* dists, hnsw_query_stats* stats, cudaStream_t s,
                          uint32_t* work, const StopModel* stop) {
    return launch_search_mode(ix, p, q, n, ids, dists, stats, s, work, stop, 0, nullptr, nullptr, nullptr);
}

// One-pass launch over an explicit device view of the index (graph
// construction and insertion search views that are not published).
hnsw_status launch_search_view(hnsw_index* ix, const DevIndex& view, const hnsw_search_params& p, const float* q,
                               uint32_t n, uint32_t* ids, float* dists, cudaStream_t s, uint32_t* work) {
    return launch_search_mode(ix, p, q, n, ids, dists, nullptr, s, work, nullptr, 0, nullptr, nullptr, nullptr,
                              nullptr, nullptr, &view);
}

// Grouped launch for the server: n queries of several requests on one index,
// per-query k/ef packed in q_kef and output offsets in q_out (device arrays),
// with max_k and max_ef sizing the per-warp state.
hnsw_status launch_search_group(hnsw_index* ix, const hnsw_search_params& p, const float* q, uint32_t n,
                                int max_k, int max_ef, const uint32_t* q_kef, const uint64_t* q_out,
                                uint32_t* ids, float* dists, cudaStream_t s, uint32_t* work,
                                const StopModel* stop) {
    hnsw_search_params pp = p;
    pp.k = max_k;
    pp.ef = max_ef;
    return launch_search_mode(ix, pp, q, n, ids, dists, nullptr, s, work, stop, 0, nullptr, nullptr, nullptr,
                              q_kef, q_out);
}

// A pair of work counters for one call (slots 2i and 2i+1 of the index's
// ring): concurrent calls on one index use different counters.
uint32_t take_work_slots(hnsw_index* ix) {
    return (ix->work_next.fetch_add(1) % uint32_t(kWorkSlots / 2)) * 2u;
}

// Reads and clears the index's error word (set by a kernel whose bounded wait
// ran out); call after the work that may set it has completed.
bool take_device_error(hnsw_index* ix) {
    if (!ix->h_err) return false;
    volatile uint32_t* w = ix->h_err;
    if (*w == 0u) return false;
    *w = 0u;
    return true;
}

// One launch over the queries of several requests of one index (the
// server's grouped dispatch); device buffers; asynchronous on s.
hnsw_status search_group(hnsw_index* ix, const hnsw_search_params& p, const float* q, uint32_t n, int max_k,
                         int max_ef, const uint32_t* q_kef, const uint64_t* q_out, uint32_t* ids, float* dists,
                         cudaStream_t s) {
    if (max_k < 1 || max_k > kMaxK || (max_ef > max_k ? max_ef : max_k) > kMaxEf)
        return fail(HNSW_EINVAL, "search group: k or ef out of range");
    if (p.rerank && !ix->dev.vec32) return fail(HNSW_EINVAL, "search group: rerank needs the fp32 copy");
    if (p.stop_period > 65535) return fail(HNSW_EINVAL, "search group: stop_period above 65535");
    StopModel sm{};
    const StopModel* smp = nullptr;
    if (p.stop_threshold > 0.0f && p.stop_threshold < 1.0f) {
        if (!ix->d_stop) return fail(HNSW_EINVAL, "search group: stop_threshold in (0,1) needs a stop model");
        sm.stop = ix->d_stop;
        sm.logit_threshold = logf(p.stop_threshold / (1.0f - p.stop_threshold));
        sm.period = p.stop_period > 0 ? p.stop_period : 8;
        smp = &sm;
    }
    return launch_search_group(ix, p, q, n, max_k, max_ef, q_kef, q_out, ids, dists, s,
                               ix->d_work + take_work_slots(ix), smp);
}

}  // namespace hnswgb

using namespace hnswgb;

extern "C" hnsw_status hnsw_search_ex(hnsw_index* ix, const hnsw_search_params* p, const float* queries, int64_t n,
                                      uint32_t* out_ids, float* out_dists, hnsw_query_stats* stats, void* stream) {
    if (!ix || !p) return fail(HNSW_EINVAL, "hnsw_search: null index or params");
    if (n < 0 || n >= (int64_t(1) << 31)) return fail(HNSW_EINVAL, "hnsw_search: n out of range");
    if (p->k < 1 || p->k > kMaxK || p->ef < 1) return fail(HNSW_EINVAL, "hnsw_search: k or ef out of range");
    if ((p->ef > p->k ? p->ef : p->k) > kMaxEf) return fail(HNSW_EINVAL, "hnsw_search: ef' above 1024");
    if (p->visited_log2 != 0 && (p->visited_log2 < 5 || p->visited_log2 > 15))
        return fail(HNSW_EINVAL, "hnsw_search: visited_log2 outside [5,15]");
    if (p->schedule < 0 || p->schedule > 3) return fail(HNSW_EINVAL, "hnsw_search: schedule outside [0,3]");
    if (p->rerank && !ix->dev.vec32) return fail(HNSW_EINVAL, "hnsw_search: rerank needs the fp32 copy");
    if (p->stop_period > 65535) return fail(HNSW_EINVAL, "hnsw_search: stop_period above 65535");
    if (n == 0) return HNSW_OK;
    if (!queries || !out_ids || !out_dists) return fail(HNSW_EINVAL, "hnsw_search: null buffer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // releases this call's hold on its stream's staging buffer on every return
    struct StageLease {
        hnsw_index* ix = nullptr;
        void* stream = nullptr;
        ~StageLease() {
            if (!ix) return;
            std::lock_guard<std::mutex> lk(ix->stage_mu);
            for (auto& st : ix->stages)
                if (st.stream == stream && st.in_use > 0) --st.in_use;
        }
    } lease;
    const bool dq = is_device_ptr(queries), di = is_device_ptr(out_ids), dd = is_device_ptr(out_dists);
    const bool ds = stats ? is_device_ptr(stats) : true;
    const size_t qb = size_t(n) * ix->dev.d * 4, ob = size_t(n) * p->k * 4, sb = stats ? size_t(n) * 16 : 0;
    const float* q = queries;
    uint32_t* ids = out_ids;
    float* dists = out_dists;
    hnsw_query_stats* st = stats;
    if (!dq || !di || !dd || !ds) {
        const size_t need = al256(qb) + 2 * al256(ob) + al256(sb);
        void* sbuf = nullptr;
        {
            // this stream's staging buffer (calls on different streams may run
            // concurrently; cudaFree synchronises the device before a buffer
            // is replaced or dropped, and only idle buffers are dropped)
            std::lock_guard<std::mutex> lk(ix->stage_mu);
            hnsw_index::Stage* e = nullptr;
            for (auto& st : ix->stages)
                if (st.stream == stream) e = &st;
            if (!e) {
                if (int(ix->stages.size()) >= kMaxStages) {
                    auto it = ix->stages.begin();
                    while (it != ix->stages.end() && it->in_use > 0) ++it;
                    if (it == ix->stages.end())
                        return fail(HNSW_EINVAL, "hnsw_search: more than 16 concurrent host-memory calls on one index");
                    if (it->buf) cudaFree(it->buf);
                    ix->stages.erase(it);
                }
                ix->stages.push_back({stream, nullptr, 0, 0});
                e = &ix->stages.back();
            }
            if (e->bytes < need) {
                if (e->buf) cudaFree(e->buf);
                e->buf = nullptr;
                e->bytes = 0;
                if (cudaMalloc(&e->buf, need) != cudaSuccess) {
                    cudaGetLastError();
                    e->buf = nullptr;
                    return fail(HNSW_ENOMEM, "hnsw_search: staging buffer");
                }
                e->bytes = need;
            }
            ++e->in_use;
            sbuf = e->buf;
        }
        lease.ix = ix;
        lease.stream = stream;
        uint8_t* sp = static_cast<uint8_t*>(sbuf);
        if (!dq) {
            q = reinterpret_cast<const float*>(sp);
            cudaError_t e = cudaMemcpyAsync(sp, queries, qb, cudaMemcpyHostToDevice, s);
            if (e != cudaSuccess) return fail(HNSW_ECUDA, std::string("hnsw_search: H2D: ") + cudaGetErrorString(e));
        }
        sp += al256(qb);
        if (!di) ids = reinterpret_cast<uint32_t*>(sp);
        sp += al256(ob);
        if (!dd) dists = reinterpret_cast<float*>(sp);
        sp += al256(ob);
        if (!ds) st = reinterpret_cast<hnsw_query_stats*>(sp);
    }
    uint32_t* work = ix->d_work + take_work_slots(ix);
    cudaError_t e = cudaSuccess;
    StopModel sm{};
    const StopModel* smp = nullptr;
    if (p->stop_threshold > 0.0f && p->stop_threshold < 1.0f) {
        if (!ix->d_stop) return fail(HNSW_EINVAL, "hnsw_search: stop_threshold in (0,1) needs a stop model");
        sm.stop = ix->d_stop;
        sm.logit_threshold = logf(p->stop_threshold / (1.0f - p->stop_threshold));
        sm.period = p->stop_period > 0 ? p->stop_period : 8;
        smp = &sm;
    }
    // schedule: 0 automatic (a block per query for small batches; deferral for
    // 33 to 2^24 queries that give some warp several; else one pass), 1 one
    // pass in input order, 2 two passes, 3 deferral
    const DevIndex snap = dev_snapshot(ix);  // both passes search the same version
    const bool two = snap.N > 0 && !p->check_bounds && p->schedule == 2;
    const Defer defer = snap.N == 0 || p->check_bounds ? Defer::no
                        : p->schedule == 3               ? Defer::always
                        : p->schedule == 0 && uint64_t(n) > kDeferWarmup && uint64_t(n) <= kDeferAutoMax
                            ? Defer::automatic
                            : Defer::no;
    hnsw_status r = HNSW_OK;
    if (!two) {
        r = launch_search_mode(ix, *p, q, uint32_t(n), ids, dists, st, s, work, smp, 0, nullptr, nullptr, nullptr,
                               nullptr, nullptr, &snap, defer);
        if (r != HNSW_OK) return r;
    } else {
        // stream-ordered scratch: enter keys [n] u64, upper counters [n][2] u32, order [n] u32
        void* scr = nullptr;
        const size_t bk = al256(size_t(n) * 8), bc = al256(size_t(n) * 8), bo = al256(size_t(n) * 4);
        keep_pool_memory();
        e = cudaMallocAsync(&scr, bk + bc + bo, s);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(HNSW_ENOMEM, "hnsw_search: scheduling scratch");
        }
        uint64_t* keys = static_cast<uint64_t*>(scr);
        uint32_t* cnt = reinterpret_cast<uint32_t*>(static_cast<char*>(scr) + bk);
        uint32_t* ord = reinterpret_cast<uint32_t*>(static_cast<char*>(scr) + bk + bc);
        r = launch_search_mode(ix, *p, q, uint32_t(n), ids, dists, st, s, work, smp, 1, keys, cnt, nullptr, nullptr,
                               nullptr, &snap);
        if (r == HNSW_OK) {
            const unsigned chunks = unsigned((uint64_t(n) + kSortChunk - 1) / kSortChunk);
            order_by_descent<<<chunks, 1024, 0, s>>>(keys, uint32_t(n), ord);
            e = cudaGetLastError();
            if (e != cudaSuccess) r = fail(HNSW_ECUDA, std::string("hnsw_search: order: ") + cudaGetErrorString(e));
        }
        if (r == HNSW_OK)
            r = launch_search_mode(ix, *p, q, uint32_t(n), ids, dists, st, s, work + 1, smp, 2, keys, cnt, ord,
                                   nullptr, nullptr, &snap);
        cudaFreeAsync(scr, s);
        if (r != HNSW_OK) return r;
    }
    if (!di || !dd || !ds) {
        if ((!di && (e = cudaMemcpyAsync(out_ids, ids, ob, cudaMemcpyDeviceToHost, s)) != cudaSuccess) ||
            (!dd && (e = cudaMemcpyAsync(out_dists, dists, ob, cudaMemcpyDeviceToHost, s)) != cudaSuccess) ||
            (!ds && (e = cudaMemcpyAsync(stats, st, sb, cudaMemcpyDeviceToHost, s)) != cudaSuccess))
            return fail(HNSW_ECUDA, std::string("hnsw_search: D2H: ") + cudaGetErrorString(e));
    }
    if (!dq || !di || !dd || !ds) {
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return fail(HNSW_ECUDA, std::string("hnsw_search: ") + cudaGetErrorString(e));
        if (take_device_error(ix))
            return fail(HNSW_ETIMEOUT, "hnsw_search: a bounded device-side wait ran out (this or an earlier call)");
    }
    return HNSW_OK;
}

extern "C" hnsw_status hnsw_debug_hold_decisions(hnsw_index* ix, int32_t on) {
    if (!ix) return fail(HNSW_EINVAL, "hnsw_debug_hold_decisions: null index");
    ix->hold_decisions.store(on ? 1 : 0);
    return HNSW_OK;
}

extern "C" hnsw_status hnsw_search(hnsw_index* ix, const float* queries, int64_t n, int32_t k, int32_t ef,
                                   uint32_t* out_ids, float* out_dists, void* stream) {
    hnsw_search_params p{};
    p.k = k;
    p.ef = ef;
    p.stop_threshold = 2.0f;
    return hnsw_search_ex(ix, &p, queries, n, out_ids, out_dists, nullptr, stream);
}

extern "C" hnsw_status hnsw_search_trace(hnsw_index* ix, const hnsw_search_params* p, const float* queries,
                                         int64_t n, int32_t max_checks, float* feats, uint32_t* topk,
                                         float* logits, int32_t* n_checks, uint32_t* out_ids, float* out_dists,
                                         hnsw_query_stats* stats, void* stream) {
    if (!ix || !p) return fail(HNSW_EINVAL, "hnsw_search_trace: null index or params");
    if (n < 0 || n >= (int64_t(1) << 31) || max_checks < 1) return fail(HNSW_EINVAL, "hnsw_search_trace: n or max_checks");
    if (p->k < 1 || p->k > kMaxK || p->ef < 1 || (p->ef > p->k ? p->ef : p->k) > kMaxEf)
        return fail(HNSW_EINVAL, "hnsw_search_trace: k or ef out of range");
    if (p->rerank && !ix->dev.vec32) return fail(HNSW_EINVAL, "hnsw_search_trace: rerank needs the fp32 copy");
    if (n == 0) return HNSW_OK;
    const void* ptrs[] = {queries, feats, topk, n_checks, out_ids, out_dists};
    for (const void* q : ptrs)
        if (!is_device_ptr(q)) return fail(HNSW_EINVAL, "hnsw_search_trace: buffers must be device memory");
    if ((logits && !is_device_ptr(logits)) || (stats && !is_device_ptr(stats)))
        return fail(HNSW_EINVAL, "hnsw_search_trace: buffers must be device memory");
    if (p->stop_period > 65535) return fail(HNSW_EINVAL, "hnsw_search_trace: stop_period above 65535");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    StopModel sm{};
    sm.stop = logits ? ix->d_stop : nullptr;
    sm.logit_threshold = 0.0f;
    sm.period = p->stop_period > 0 ? p->stop_period : 4;
    sm.tr_feat = feats;
    sm.tr_topk = topk;
    sm.tr_logit = ix->d_stop ? logits : nullptr;
    sm.tr_count = n_checks;
    sm.tr_max = max_checks;
    uint32_t* work = ix->d_work + take_work_slots(ix);
    hnsw_search_params q = *p;
    return launch_search(ix, q, queries, uint32_t(n), out_ids, out_dists, stats, s, work, &sm);
}
