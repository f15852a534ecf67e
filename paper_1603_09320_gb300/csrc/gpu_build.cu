// gpu_build.cu -- bulk construction of the graph with the insertions of
// layer-0 elements done on the GPU in batches (Alg. 1 with Alg. 4 as
// SELECT-NEIGHBORS; parallel construction, Section 4.1).
//
// Decomposition.  On layers >= 1, Alg. 1 only involves elements whose level
// is >= 1: a search on layer lc >= 1 visits only elements present there, and
// only they receive links there.  So the graph is built in two parts:
//  1. a seed set -- every element of level >= 1 plus the first elements of
//     the data -- inserted in id order on the host (hnsw_build), which gives
//     the upper layers and the seed's layer-0 links;
//  2. the remaining elements (all of level 0) inserted into layer 0 on the
//     GPU in batches, in id order: for a batch, every element searches the
//     graph as it stands before the batch (Alg. 5's descent through the upper
//     layers, then SEARCH-LAYER with ef = efConstruction on layer 0, run by the
//     library's search kernel), selects its M links (Alg. 4's selection), and
//     the reverse links are added per target element, which shrinks its list
//     with Alg. 4 when it exceeds Mmax0 (Alg. 1's reverse links and shrink).
// Elements of one batch do not see one another (they are linked only through
// the elements they link to); a batch is at most 1/16 of the elements already
// inserted, so each element searches a graph that already holds at least 94%
// of what precedes it.  The insertion order is a permutation of Alg. 1's (seed
// first) with batch-parallel semantics, so the graph is not the sequential
// one; it is deterministic, and on integer data equal byte for byte to the
// oracle's batch form of Alg. 1 (which batches of one element reduce to
// Alg. 1 itself).
#include <cub/cub.cuh>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "common.hpp"
#include "index.cuh"

namespace hnswgb {
// defined in search.cu
hnsw_status launch_search_view(hnsw_index* ix, const DevIndex& view, const hnsw_search_params& p, const float* q,
                               uint32_t n, uint32_t* ids, float* dists, cudaStream_t s, uint32_t* work);
}  // namespace hnswgb

namespace {

using namespace hnswgb;

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxDW = 8;      // coordinates per lane: d <= 256
constexpr int kChunk = 64;     // candidates a selection looks at together
constexpr int kKeep = 256;     // shrink candidates examined per chunk (ascending key order)
constexpr int kKeyBuf = 512;   // candidate keys sorted at once in a shrink
constexpr int kMaxOld = 64;    // members of a list (Mmax0, Mmax <= 64)
constexpr int kWarps = 4;      // warps per block of the selection kernels

__device__ __forceinline__ uint32_t f2ord(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t o) {
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// Shared memory of one warp's selection.
struct SelSmem {
    uint32_t cid[kChunk];   // the chunk's candidates
    float cd[kChunk];
    uint32_t live[kChunk];  // indexes of those not rejected yet, in order
    uint32_t keep[kChunk];
    uint32_t Rid[kMaxOld];  // accepted elements and their distances to the base
    float Rd[kMaxOld];
    uint32_t Did[kMaxOld];  // the first discarded candidates, in order (keepPrunedConnections)
    float Dd[kMaxOld];
};

// A row in the registers of a team of 8 lanes: lane t holds the 16-byte chunks
// t, t + 8, ... (coordinates 4t .. 4t+3 of every 32).
// DW: 32-coordinate pieces per row (4: d <= 128, 8: d <= 256).
template <int DW>
struct TeamVec {
    float4 v[DW];
};
template <int DW>
__device__ __forceinline__ void load_team(const float* rows, uint32_t stride, uint32_t id, TeamVec<DW>& x, int lane) {
    const float4* r = reinterpret_cast<const float4*>(rows + uint64_t(id) * stride);
#pragma unroll
    for (int k = 0; k < DW; ++k) {
        const uint32_t c = uint32_t(8 * k + (lane & 7));
        x.v[k] = 32u * k < stride && 4u * c < stride ? __ldg(r + c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
}

// Distance between x and y, in every lane of the team.  The sum of coordinates
// c = l (mod 32) is formed first, for every l, and these 32 sums are added as
// a butterfly over l would (16, 8, 4, 2, 1 apart): steps 16, 8 and 4 go across
// lanes, with half of the sums handed over at each, 2 and 1 across what the
// lanes then hold.
template <int DW>
__device__ __forceinline__ float dist_team(const TeamVec<DW>& x, const TeamVec<DW>& y, int metric, int lane) {
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < DW; ++k) {  // pieces beyond the row are zero in both and add nothing
        const float a[4] = {x.v[k].x, x.v[k].y, x.v[k].z, x.v[k].w}, b[4] = {y.v[k].x, y.v[k].y, y.v[k].z, y.v[k].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (metric == HNSW_L2SQ) {
                const float t = a[i] - b[i];
                s[i] = fmaf(t, t, s[i]);
            } else {
                s[i] = fmaf(a[i], b[i], s[i]);
            }
        }
    }
    const bool h4 = lane & 4, h2 = lane & 2;
    const float u0 = (h4 ? s[2] : s[0]) + __shfl_xor_sync(kFull, h4 ? s[0] : s[2], 4);
    const float u1 = (h4 ? s[3] : s[1]) + __shfl_xor_sync(kFull, h4 ? s[1] : s[3], 4);
    float v = (h2 ? u1 : u0) + __shfl_xor_sync(kFull, h2 ? u0 : u1, 2);
    v += __shfl_xor_sync(kFull, v, 1);
    v += __shfl_xor_sync(kFull, v, 4);
    v += __shfl_xor_sync(kFull, v, 2);
    return metric == HNSW_L2SQ ? v : 1.0f - v;
}

// Drops from the live candidates those that are not closer to the base than
// to element r (strictly; Alg. 4's test); returns how many remain.
template <int DW>
__device__ int prune(const float* rows, uint32_t stride, int metric, uint32_t r, SelSmem& w, int na, int lane) {
    TeamVec<DW> x;
    load_team(rows, stride, r, x, lane);
    const int team = lane >> 3;
    for (int base = 0; base < na; base += 8) {  // two rows per team in flight
        const int j0 = min(base + team, na - 1), j1 = min(base + 4 + team, na - 1);
        const uint32_t i0 = w.live[j0], i1 = w.live[j1];
        TeamVec<DW> y0, y1;
        load_team(rows, stride, w.cid[i0], y0, lane);
        load_team(rows, stride, w.cid[i1], y1, lane);
        const float d0 = dist_team(x, y0, metric, lane), d1 = dist_team(x, y1, metric, lane);
        if ((lane & 7) == 0) {
            w.keep[j0] = w.cd[i0] < d0;
            w.keep[j1] = w.cd[i1] < d1;
        }
    }
    __syncwarp();
    const bool k0 = lane < na && w.keep[lane], k1 = lane + 32 < na && w.keep[lane + 32];
    const uint32_t v0 = k0 ? w.live[lane] : 0u, v1 = k1 ? w.live[lane + 32] : 0u;
    const unsigned m0 = __ballot_sync(kFull, k0), m1 = __ballot_sync(kFull, k1), below = (1u << lane) - 1u;
    __syncwarp();  // every lane has read its entries before any is overwritten (a ballot orders no memory)
    if (k0) w.live[__popc(m0 & below)] = v0;
    if (k1) w.live[__popc(m0) + __popc(m1 & below)] = v1;
    __syncwarp();
    return __popc(m0) + __popc(m1);
}

// SELECT-NEIGHBORS, resumable: takes the nc <= kChunk candidates in w.cid /
// w.cd, sorted by (distance to the base, id) and following every candidate of
// earlier calls, into R (w.Rid / Rd; nr entries so far), at most cap.
// heuristic: Alg. 4's acceptance loop without extendCandidates (a candidate is
// accepted when it is closer to the base than to every element accepted
// before it, strictly); the discarded ones are recorded in order (nd so far,
// the first cap of them: keepPrunedConnections never takes more).  Otherwise
// Alg. 3 (the cap nearest).
// Alg. 4 asks of each candidate in turn whether an accepted element rejects
// it; here each accepted element, in turn, rejects candidates: the next to be
// accepted is the first one left, and the elements it is tested against are
// those accepted before it, as in the loop.  A rejection step scores its
// candidates 4 at a time (8 lanes each) instead of one after another, each
// waiting for the last; a chain of at most cap steps per chunk.  Measured on
// 1,000 elements into 20,000 (128 coordinates, efConstruction 200): a batch's
// select_forward took 241 us and takes 97, its link_reverse 239 and 88.
template <int DW>
__device__ void select_more(const float* rows, uint32_t stride, int metric, int nc, int cap, bool heuristic,
                            SelSmem& w, int& nr, int& nd, int lane) {
    if (!heuristic) {
        const int take = min(nc, cap - nr);
        for (int i = lane; i < take; i += 32) {
            w.Rid[nr + i] = w.cid[i];
            w.Rd[nr + i] = w.cd[i];
        }
        nr += take;
        __syncwarp();
        return;
    }
    for (int i = lane; i < nc; i += 32) w.live[i] = uint32_t(i);
    __syncwarp();
    int na = nc;
    for (int j = 0; j < nr && na > 0; ++j) na = prune<DW>(rows, stride, metric, w.Rid[j], w, na, lane);
    uint64_t taken = 0;  // accepted in this chunk
    while (na > 0 && nr < cap) {
        const uint32_t i = w.live[0];
        const uint32_t r = w.cid[i];
        if (lane == 0) {
            w.Rid[nr] = r;
            w.Rd[nr] = w.cd[i];
        }
        taken |= 1ull << i;
        ++nr;
        __syncwarp();
        // the rest of the list, without r itself
        const uint32_t v0 = lane + 1 < na ? w.live[lane + 1] : 0u, v1 = lane + 33 < na ? w.live[lane + 33] : 0u;
        __syncwarp();
        if (lane + 1 < na) w.live[lane] = v0;
        if (lane + 33 < na) w.live[lane + 32] = v1;
        __syncwarp();
        if (--na > 0 && nr < cap) na = prune<DW>(rows, stride, metric, r, w, na, lane);
    }
    for (int h = 0; h < nc; h += 32) {
        const int i = h + lane;
        const bool out = i < nc && !((taken >> i) & 1ull);
        const unsigned m = __ballot_sync(kFull, out);
        const int p = nd + __popc(m & ((1u << lane) - 1u));
        if (out && p < cap) {
            w.Did[p] = w.cid[i];
            w.Dd[p] = w.cd[i];
        }
        nd = min(cap, nd + __popc(m));
    }
    __syncwarp();
}

// Alg. 4's last step (keepPrunedConnections): the nearest discarded
// candidates fill R up to cap.
__device__ void append_pruned(SelSmem& w, int cap, int& nr, int nd, int lane) {
    const int take = min(nd, cap - nr);
    for (int i = lane; i < take; i += 32) {
        w.Rid[nr + i] = w.Did[i];
        w.Rd[nr + i] = w.Dd[i];
    }
    nr += max(take, 0);
    __syncwarp();
}

// SELECT-NEIGHBORS over a sorted candidate list (element i given by get(i, id,
// distance)); returns |R|.
template <int DW, class Get>
__device__ __forceinline__ int select_links(const float* rows, uint32_t stride, int metric, Get get, int nc, int cap,
                                            bool heuristic, bool keep_pruned, SelSmem& w, int lane) {
    int nr = 0, nd = 0;
    for (int base = 0; base < nc && nr < cap; base += kChunk) {
        const int m = min(kChunk, nc - base);
        for (int i = lane; i < m; i += 32) get(base + i, w.cid[i], w.cd[i]);
        __syncwarp();
        select_more<DW>(rows, stride, metric, m, cap, heuristic, w, nr, nd, lane);
    }
    if (heuristic && keep_pruned) append_pruned(w, cap, nr, nd, lane);
    return nr;
}

__global__ void gather_rows(const float* __restrict__ rows, uint32_t stride, uint32_t d,
                            const uint32_t* __restrict__ ids, uint32_t n, float* __restrict__ out) {
    const uint64_t t = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= uint64_t(n) * d) return;
    const uint32_t j = uint32_t(t / d), c = uint32_t(t % d);
    out[t] = rows[uint64_t(ids[j]) * stride + c];
}

// One warp per new element b: its M links from its search result (sorted
// (dist, id), kNone-padded), written to its layer-0 row, and one reverse
// pair per link: key = the linked element, value = the new element and their
// distance (pairs of unused slots get key kNone).
template <int DW>
__global__ void __launch_bounds__(kWarps * 32) select_forward(
    const float* __restrict__ rows, uint32_t stride, int metric, const uint32_t* __restrict__ bids, uint32_t B, const uint32_t* __restrict__ res_id,
    const float* __restrict__ res_d, int efc, int M, int heuristic, int keep_pruned, uint32_t* __restrict__ nbr0,
    uint32_t s0, uint32_t* __restrict__ pkey, uint32_t* __restrict__ pval, float* __restrict__ pdist) {
    __shared__ SelSmem sel[kWarps];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint32_t b = blockIdx.x * kWarps + wib;
    if (b >= B) return;
    SelSmem& w = sel[wib];
    const uint32_t q = bids[b];
    const uint32_t* cid = res_id + uint64_t(b) * efc;
    const float* cd = res_d + uint64_t(b) * efc;
    int nc = 0;
    for (int i = lane; i < efc; i += 32) nc += cid[i] != kNone && cid[i] != q;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nc += __shfl_xor_sync(kFull, nc, o);
    // results are sorted with the kNone padding last; q itself is never reachable
    const int nr = select_links<DW>(
        rows, stride, metric,
        [&](int i, uint32_t& id, float& dist) {
            id = cid[i];
            dist = cd[i];
        },
        nc, M, heuristic != 0, keep_pruned != 0, w, lane);
    for (int j = lane; j < M; j += 32) {
        const uint64_t o = uint64_t(b) * M + j;
        if (j < nr) {
            nbr0[uint64_t(q) * s0 + j] = w.Rid[j];
            pkey[o] = w.Rid[j];
            pval[o] = q;
            pdist[o] = w.Rd[j];
        } else {
            pkey[o] = kNone;
            pval[o] = kNone;
            pdist[o] = 0.0f;
        }
    }
}

__global__ void mark_segments(const uint32_t* __restrict__ skey, uint32_t n, uint32_t* __restrict__ seg,
                              uint32_t* __restrict__ nseg) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t k = skey[i];
    if (k != kNone && (i == 0 || skey[i - 1] != k)) seg[atomicAdd(nseg, 1u)] = i;
}

// warp bitonic sort of n keys (power of two) in shared memory, ascending
__device__ void sort_keys(uint64_t* a, int n, int lane) {
    for (int kk = 2; kk <= n; kk <<= 1)
        for (int j = kk >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < n; i += 32) {
                const int p = i ^ j;
                if (p > i) {
                    const uint64_t x = a[i], y = a[p];
                    if ((x > y) == ((i & kk) == 0)) {
                        a[i] = y;
                        a[p] = x;
                    }
                }
            }
            __syncwarp();
        }
}

__device__ __forceinline__ unsigned lanes_below(int lane) { return (1u << lane) - 1u; }

// One warp per target element e (a segment of the sorted pairs): the new
// elements linking to e join neighbourhood(e); when the list then exceeds
// Mmax0 it becomes SELECT-NEIGHBORS(e, eConn, Mmax0) over all of eConn, the
// current members and the new ones (Alg. 1's reverse links and shrink).  Alg. 4 takes eConn
// in ascending (distance, id) order and stops once Mmax0 are accepted; here
// that order is walked in chunks of kKeep: each chunk is the kKeep smallest
// keys above the previous chunk's last one (keys are distinct: ids are),
// found by one pass over the candidates that sorts kKeyBuf keys at a time.
template <int DW>
__global__ void __launch_bounds__(kWarps * 32) link_reverse(
    const float* __restrict__ rows, uint32_t stride, int metric, const uint32_t* __restrict__ skey,
    const uint32_t* __restrict__ sidx, uint32_t npairs,
    const uint32_t* __restrict__ seg, const uint32_t* __restrict__ nseg, const uint32_t* __restrict__ pval,
    const float* __restrict__ pdist, uint32_t* __restrict__ nbr0, uint32_t s0, int Mmax0, int heuristic,
    int keep_pruned) {
    __shared__ SelSmem sel[kWarps];
    __shared__ uint64_t key_buf[kWarps][kKeyBuf];
    __shared__ uint64_t old_keys[kWarps][kMaxOld];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nw = kWarps;
    SelSmem& w = sel[wib];
    uint64_t* keys = key_buf[wib];    // shrink candidates, (ordered distance, id)
    uint64_t* okeys = old_keys[wib];  // keys of the list's current members
    const uint32_t nsegs = *nseg;
    for (uint32_t s = blockIdx.x * nw + wib; s < nsegs; s += gridDim.x * nw) {
        const uint32_t i0 = seg[s];
        const uint32_t e = skey[i0];
        uint32_t i1 = i0 + 1;
        while (i1 < npairs && skey[i1] == e) ++i1;  // segments are short
        uint32_t* row = nbr0 + uint64_t(e) * s0;
        int n0 = 0;
        for (int j = lane; j < Mmax0; j += 32) n0 += row[j] != kNone;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) n0 += __shfl_xor_sync(kFull, n0, o);
        const int nin = int(i1 - i0);
        if (n0 + nin <= Mmax0) {  // room: append in insertion order
            for (int t = lane; t < nin; t += 32) row[n0 + t] = pval[sidx[i0 + t]];
            __syncwarp();
            continue;
        }
        // keys of the current members (their distances to e recomputed)
        {
            TeamVec<DW> x;
            load_team(rows, stride, e, x, lane);
            for (int j0 = 0; j0 < n0; j0 += 4) {
                const int j = min(j0 + (lane >> 3), n0 - 1);
                const uint32_t c = row[j];
                TeamVec<DW> y;
                load_team(rows, stride, c, y, lane);
                const float dc = dist_team(x, y, metric, lane);
                if ((lane & 7) == 0) okeys[j] = (uint64_t(f2ord(dc)) << 32) | c;
            }
        }
        __syncwarp();
        const int total = n0 + nin;
        int nr = 0, nd = 0, seen = 0;
        uint64_t last = 0;  // keys of the next chunk are above it (all keys in the first chunk)
        bool first = true;
        for (;;) {
            // the kKeep smallest candidate keys above `last`
            int nk = 0;
            for (int b0 = 0; b0 < total; b0 += 32) {
                const int j = b0 + lane;
                uint64_t k = ~0ull;
                if (j < n0) {
                    k = okeys[j];
                } else if (j < total) {
                    const uint32_t pi = sidx[i0 + uint32_t(j - n0)];
                    k = (uint64_t(f2ord(pdist[pi])) << 32) | pval[pi];
                }
                const bool ok = j < total && (first || k > last);
                const unsigned m = __ballot_sync(kFull, ok);
                if (ok) keys[nk + __popc(m & lanes_below(lane))] = k;
                nk += __popc(m);
                if (nk > kKeyBuf - 32) {  // full: keep the kKeep smallest
                    for (int u = nk + lane; u < kKeyBuf; u += 32) keys[u] = ~0ull;
                    __syncwarp();
                    sort_keys(keys, kKeyBuf, lane);
                    nk = kKeep;
                }
                __syncwarp();
            }
            int n2 = 32;
            while (n2 < nk) n2 <<= 1;
            for (int u = nk + lane; u < n2; u += 32) keys[u] = ~0ull;
            __syncwarp();
            sort_keys(keys, n2, lane);
            nk = min(nk, kKeep);
            if (nk == 0) break;
            for (int base = 0; base < nk && nr < Mmax0; base += kChunk) {
                const int m = min(kChunk, nk - base);
                for (int i = lane; i < m; i += 32) {
                    w.cid[i] = uint32_t(keys[base + i] & 0xffffffffu);
                    w.cd[i] = ord2f(uint32_t(keys[base + i] >> 32));
                }
                __syncwarp();
                select_more<DW>(rows, stride, metric, m, Mmax0, heuristic != 0, w, nr, nd, lane);
            }
            seen += nk;
            if (nr >= Mmax0 || seen >= total) break;
            last = keys[nk - 1];
            first = false;
            __syncwarp();
        }
        if (heuristic && keep_pruned) append_pruned(w, Mmax0, nr, nd, lane);
        for (int j = lane; j < Mmax0; j += 32) row[j] = j < nr ? w.Rid[j] : kNone;
        __syncwarp();
    }
}

struct DevBuf {
    void* p = nullptr;
    ~DevBuf() {
        if (p) cudaFree(p);
    }
};

hnsw_status cuda_fail(cudaError_t e, const char* what) {
    return fail(HNSW_ECUDA, std::string("hnsw_build_gpu: ") + what + ": " + cudaGetErrorString(e));
}

}  // namespace

namespace hnswgb {

// Inserts the elements `ids` (in order, all of level 0 or already linked on
// their upper layers) into layer 0 of `view` in batches of at most 1/16 of
// the elements inserted so far (`inserted` before the first batch), on
// stream s.  The view's rows must be fp32 (storage F32) and its nbr0 is the
// adjacency written; asynchronous, buffers freed at return (cudaFree waits
// for the stream's work).
hnsw_status insert_layer0(hnsw_index* ix, const DevIndex& view, const std::vector<uint32_t>& ids, uint64_t inserted,
                          int metric, int M, int Mmax0, int efc, int heuristic, int keep_pruned, cudaStream_t s) {
    if (ids.empty()) return HNSW_OK;
    const DevIndex& D = view;
    const float* drows = reinterpret_cast<const float*>(D.vec);
    const uint32_t d = D.d, stride = D.row_chunks * 4, s0 = D.s0;
    uint32_t* nbr0 = const_cast<uint32_t*>(D.nbr0);
    const uint32_t Bmax = uint32_t(std::min<uint64_t>(32768, std::max<uint64_t>(64, ids.size())));
    DevBuf dbid, dq, rid, rdist, pkey, pval, pdist, skey, sidx, idx, seg, nseg, work, tmp;
    size_t tmp_bytes = 0;
    const uint32_t npair_max = Bmax * uint32_t(M);
    cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, static_cast<uint32_t*>(nullptr),
                                    static_cast<uint32_t*>(nullptr), static_cast<uint32_t*>(nullptr),
                                    static_cast<uint32_t*>(nullptr), int(npair_max), 0, 32, s);
    cudaError_t e = cudaSuccess;
    auto alloc = [&](DevBuf& x, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(&x.p, bytes ? bytes : 16);
    };
    alloc(dbid, size_t(ids.size()) * 4);
    alloc(dq, size_t(Bmax) * d * 4);
    alloc(rid, size_t(Bmax) * efc * 4);
    alloc(rdist, size_t(Bmax) * efc * 4);
    alloc(pkey, size_t(npair_max) * 4);
    alloc(pval, size_t(npair_max) * 4);
    alloc(pdist, size_t(npair_max) * 4);
    alloc(skey, size_t(npair_max) * 4);
    alloc(sidx, size_t(npair_max) * 4);
    alloc(idx, size_t(npair_max) * 4);
    alloc(seg, size_t(npair_max) * 4);
    alloc(nseg, 16);
    alloc(work, 16);
    alloc(tmp, tmp_bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(HNSW_ENOMEM, "layer-0 insertion: device buffers");
    }
    std::vector<uint32_t> iota(npair_max);
    for (uint32_t i = 0; i < npair_max; ++i) iota[i] = i;
    // pageable sources: the copies complete before cudaMemcpyAsync returns
    if ((e = cudaMemcpyAsync(idx.p, iota.data(), size_t(npair_max) * 4, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(dbid.p, ids.data(), ids.size() * 4, cudaMemcpyHostToDevice, s)) != cudaSuccess)
        return cuda_fail(e, "copy");
    const bool wide = stride > 128;
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    hnsw_search_params sp{};
    sp.k = efc;
    sp.ef = efc;
    hnsw_status st = HNSW_OK;
    for (size_t pos = 0; pos < ids.size();) {
        const uint32_t B = uint32_t(std::min<uint64_t>(
            {uint64_t(Bmax), uint64_t(ids.size() - pos), std::max<uint64_t>(64, inserted / 16)}));
        const uint32_t* bids = static_cast<const uint32_t*>(dbid.p) + pos;
        const uint64_t nq = uint64_t(B) * d;
        gather_rows<<<unsigned((nq + 255) / 256), 256, 0, s>>>(drows, stride, d, bids, B, static_cast<float*>(dq.p));
        st = launch_search_view(ix, view, sp, static_cast<const float*>(dq.p), B, static_cast<uint32_t*>(rid.p),
                                static_cast<float*>(rdist.p), s, static_cast<uint32_t*>(work.p));
        if (st != HNSW_OK) break;
        (wide ? select_forward<8> : select_forward<4>)<<<(B + kWarps - 1) / kWarps, kWarps * 32, 0, s>>>(
            drows, stride, metric, bids, B, static_cast<const uint32_t*>(rid.p),
            static_cast<const float*>(rdist.p), efc, M, heuristic, keep_pruned, nbr0, s0,
            static_cast<uint32_t*>(pkey.p), static_cast<uint32_t*>(pval.p), static_cast<float*>(pdist.p));
        const uint32_t np = B * uint32_t(M);
        size_t tb = tmp_bytes;
        if ((e = cub::DeviceRadixSort::SortPairs(tmp.p, tb, static_cast<const uint32_t*>(pkey.p),
                                                 static_cast<uint32_t*>(skey.p), static_cast<const uint32_t*>(idx.p),
                                                 static_cast<uint32_t*>(sidx.p), int(np), 0, 32, s)) != cudaSuccess)
            break;
        if ((e = cudaMemsetAsync(nseg.p, 0, 4, s)) != cudaSuccess) break;
        mark_segments<<<(np + 255) / 256, 256, 0, s>>>(static_cast<const uint32_t*>(skey.p), np,
                                                      static_cast<uint32_t*>(seg.p), static_cast<uint32_t*>(nseg.p));
        (wide ? link_reverse<8> : link_reverse<4>)<<<unsigned(sms) * 4, kWarps * 32, 0, s>>>(
            drows, stride, metric, static_cast<const uint32_t*>(skey.p), static_cast<const uint32_t*>(sidx.p),
            np, static_cast<const uint32_t*>(seg.p), static_cast<const uint32_t*>(nseg.p),
            static_cast<const uint32_t*>(pval.p), static_cast<const float*>(pdist.p), nbr0, s0, Mmax0, heuristic,
            keep_pruned);
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        pos += B;
        inserted += B;
    }
    if (st != HNSW_OK) return st;
    if (e != cudaSuccess) return cuda_fail(e, "batch");
    return HNSW_OK;
}

}  // namespace hnswgb

extern "C" hnsw_status hnsw_build_gpu(const float* data, uint64_t N, uint32_t d, hnsw_metric metric,
                                      const hnsw_build_params* params, const double* level_u, void* stream,
                                      void** out_blob, uint64_t* out_bytes) {
    if (!params || !out_blob || !out_bytes || (N > 0 && (!data || !level_u)))
        return fail(HNSW_EINVAL, "hnsw_build_gpu: null pointer");
    const hnsw_build_params& p = *params;
    if (d == 0 || d > 32u * kMaxDW || N >= (1ull << 31) || p.M == 0 || p.M > p.Mmax || p.M > p.Mmax0 ||
        p.Mmax0 > 64 || p.Mmax > 64 || !(p.mL > 0) || p.ef_construction == 0 || p.ef_construction > 1024 ||
        p.extend_candidates || (metric != HNSW_L2SQ && metric != HNSW_COSINE))
        return fail(HNSW_EINVAL, "hnsw_build_gpu: invalid parameters (d <= 256, efConstruction <= 1024, "
                                 "no extendCandidates)");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // levels (the level draw of Alg. 1) and the seed: the first elements and every
    // element of level >= 1, in id order
    std::vector<uint8_t> level(N);
    uint64_t rows = 0;
    for (uint64_t i = 0; i < N; ++i) {
        const double u = level_u[i];
        if (!(u > 0.0 && u <= 1.0)) return fail(HNSW_EINVAL, "hnsw_build_gpu: level_u outside (0,1]");
        const double lv = std::floor(-std::log(u) * p.mL);
        if (lv > 255) return fail(HNSW_EINVAL, "hnsw_build_gpu: level above 255");
        level[i] = uint8_t(lv);
        rows += level[i];
    }
    const uint64_t n_first = std::min<uint64_t>(N, 4096);
    std::vector<uint32_t> seed, rest;
    for (uint64_t i = 0; i < N; ++i) (i < n_first || level[i] > 0 ? seed : rest).push_back(uint32_t(i));
    if (rest.empty()) return hnsw_build(data, N, d, metric, params, level_u, out_blob, out_bytes);
    // 1. the seed on the host
    std::vector<float> sdata(seed.size() * size_t(d));
    std::vector<double> su(seed.size());
    for (size_t j = 0; j < seed.size(); ++j) {
        std::memcpy(&sdata[j * d], data + uint64_t(seed[j]) * d, d * 4ull);
        su[j] = level_u[seed[j]];
    }
    void* sblob = nullptr;
    uint64_t sbytes = 0;
    hnsw_status st = hnsw_build(sdata.data(), seed.size(), d, metric, params, su.data(), &sblob, &sbytes);
    if (st != HNSW_OK) return st;
    BlobHeader sh{};
    read_header(static_cast<const uint8_t*>(sblob), sbytes, sh);
    const BlobLayout sl = BlobLayout::of(seed.size(), d, p.Mmax0, p.Mmax, sh.n_upper_rows);
    // the full blob: all vectors and levels, the seed's links in original ids
    const BlobLayout lay = BlobLayout::of(N, d, p.Mmax0, p.Mmax, rows);
    uint8_t* b = static_cast<uint8_t*>(std::calloc(lay.total, 1));
    if (!b) {
        hnsw_free_blob(sblob);
        return fail(HNSW_ENOMEM, "hnsw_build_gpu: blob allocation failed");
    }
    const uint8_t* sb = static_cast<const uint8_t*>(sblob);
    std::memcpy(b + lay.data, data, N * d * 4ull);
    std::memcpy(b + lay.level, level.data(), N);
    std::memset(b + lay.nbr0, 0xFF, N * p.Mmax0 * 4ull);  // every slot kNone
    auto map = [&](uint32_t v) { return v == kNone ? kNone : seed[v]; };
    for (size_t j = 0; j < seed.size(); ++j)
        for (uint32_t c = 0; c < p.Mmax0; ++c)
            wr<uint32_t>(b + lay.nbr0 + (uint64_t(seed[j]) * p.Mmax0 + c) * 4,
                         map(rd<uint32_t>(sb + sl.nbr0 + (uint64_t(j) * p.Mmax0 + c) * 4)));
    // upper rows are element-major; the seed holds every element of level >= 1
    // in id order, so its rows are already in the full graph's order
    for (uint64_t r = 0; r < sh.n_upper_rows * p.Mmax; ++r)
        wr<uint32_t>(b + lay.nbrU + r * 4, map(rd<uint32_t>(sb + sl.nbrU + r * 4)));
    BlobHeader h = sh;
    h.N = N;
    h.ep = map(sh.ep);
    h.n_upper_rows = rows;
    hnsw_free_blob(sblob);
    auto finish_header = [&]() {
        h.checksum = checksum64(b + 128, lay.total - 128, s);
        write_header(b, h);
    };
    // 2. layer-0 insertion of the rest on the GPU (the intermediate blob is
    // uploaded without its checksum or per-list checks: written just above)
    h.checksum = 0;
    write_header(b, h);
    hnsw_index* ix = nullptr;
    st = upload_index(b, lay.total, HNSW_F32, 0, stream, &ix, true);
    if (st != HNSW_OK) {
        std::free(b);
        return st;
    }
    struct IxGuard {
        hnsw_index* ix;
        ~IxGuard() { hnsw_free_index(ix); }
    } ixg{ix};
    st = insert_layer0(ix, ix->dev, rest, seed.size(), int(metric), int(p.M), int(p.Mmax0),
                       int(p.ef_construction), p.heuristic, p.keep_pruned, s);
    if (st != HNSW_OK) {
        std::free(b);
        return st;
    }
    uint32_t* nbr0 = static_cast<uint32_t*>(ix->d_nbr0);
    const uint32_t s0 = ix->dev.s0;
    cudaError_t e = cudaSuccess;
    // 3. the final layer 0 back into the blob
    std::vector<uint32_t> h0(N * size_t(s0));
    if ((e = cudaMemcpyAsync(h0.data(), nbr0, h0.size() * 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess) {
        std::free(b);
        return cuda_fail(e, "layer 0 copy");
    }
    for (uint64_t i = 0; i < N; ++i)
        for (uint32_t c = 0; c < p.Mmax0; ++c) wr<uint32_t>(b + lay.nbr0 + (i * p.Mmax0 + c) * 4, h0[i * s0 + c]);
    finish_header();
    *out_blob = b;
    *out_bytes = lay.total;
    return HNSW_OK;
}

// ---------------------------------------------------------------------------
// Incremental insertion into a resident index
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ uint64_t mkkey(float d, uint32_t id) { return (uint64_t(f2ord(d)) << 32) | id; }
__device__ __forceinline__ uint32_t kid(uint64_t k) { return uint32_t(k & 0xffffffffu); }
__device__ __forceinline__ float kdist(uint64_t k) { return ord2f(uint32_t(k >> 32)); }

// keys of the single-list search: (ordered distance, id, expanded bit)
__device__ __forceinline__ uint32_t lid(uint64_t k) { return uint32_t(k >> 1) & 0x7fffffffu; }

struct UpperArgs {
    DevIndex v;                 // fp32 view; nbrU / upoff of the version being written
    const uint32_t* ids;        // new elements of level >= 1, in id order
    const uint8_t* lv;          // their levels
    uint32_t n;
    int efc, M, Mmax, heuristic, keep_pruned;
    uint32_t* visited;          // [capacity] epoch tags
    int* state;                 // {enter point, top level}
};

__device__ __forceinline__ uint32_t* upper_row(const UpperArgs& a, uint32_t e, int lc) {
    return const_cast<uint32_t*>(a.v.nbrU) + (uint64_t(a.v.upoff[e]) + uint32_t(lc - 1)) * a.v.sU;
}

constexpr int kUpWarps = 16;
constexpr int kUpThreads = kUpWarps * 32;

// E * kUpThreads entries of W
template <int E>
struct UpperSmem {
    uint64_t T[2][E * kUpThreads];  // W, and the W that the next merge makes
    uint64_t Ek[E * kUpThreads];    // enter points of a layer's search, sorted; afterwards its result
    uint64_t K[2][kMaxOld];         // an expansion's new keys (all ones: none), two expansions' worth
    uint32_t ids[2][kMaxOld];       // and its neighbours
    uint64_t best[2][kUpWarps];     // descent: each warp's best neighbour (two steps' worth)
    int first;                      // where the smallest new key went
    uint32_t qR[kMaxOld];         // the new element's links
    int nr;
    SelSmem sel[kUpWarps];
    uint64_t keys[kUpWarps][2 * kMaxOld];  // a reverse link's members, sorted
    float4 q[8 * kMaxDW];                  // the new element
    float4 t[kUpWarps][8 * kMaxDW];        // each warp's row (dist_seq, dist_lane)
};

// A row in the registers of a warp (lane l: chunks l and l + 32 of 4 coordinates).
template <int DW>
__device__ __forceinline__ void load_warp(float4 (&v)[DW / 4], const float* rows, uint32_t stride, uint32_t id, int lane) {
    const float4* r = reinterpret_cast<const float4*>(rows + uint64_t(id) * stride);
#pragma unroll
    for (int k = 0; k < DW / 4; ++k) {
        const uint32_t c = uint32_t(lane + 32 * k);
        v[k] = 4u * c < stride ? __ldg(r + c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
}
// Distance between q (shared memory, stride floats) and such a row, in every
// lane, the coordinates added one after another: the order in which the upper
// layers have always been scored (near-ties decide links).  The warp's lanes
// hold four coordinates each, so the row goes through t (the warp's shared
// memory, 8 DW chunks), which every lane then reads from its start.
template <int DW>
__device__ __forceinline__ float dist_seq(const float4* q, const float4 (&v)[DW / 4], uint32_t stride, int metric,
                                          float4* t, int lane) {
    const bool l2 = metric == HNSW_L2SQ;
    __syncwarp();  // the previous row is read
#pragma unroll
    for (int k = 0; k < DW / 4; ++k) {
        const int c = lane + 32 * k;
        if (4u * c < stride) {
            const float4 a = q[c];
            t[c] = l2 ? make_float4(a.x - v[k].x, a.y - v[k].y, a.z - v[k].z, a.w - v[k].w) : v[k];
        }
    }
    __syncwarp();
    float s = 0.0f;
    if (l2) {
#pragma unroll 8
        for (uint32_t c = 0; 4u * c < stride; ++c) {
            const float4 a = t[c];
            s = fmaf(a.x, a.x, s);
            s = fmaf(a.y, a.y, s);
            s = fmaf(a.z, a.z, s);
            s = fmaf(a.w, a.w, s);
        }
        return s;
    }
#pragma unroll 4
    for (uint32_t c = 0; 4u * c < stride; ++c) {
        const float4 a = q[c], b = t[c];
        s = fmaf(a.x, b.x, s);
        s = fmaf(a.y, b.y, s);
        s = fmaf(a.z, b.z, s);
        s = fmaf(a.w, b.w, s);
    }
    return 1.0f - s;
}
// The same for row `id`, by one lane.
__device__ __forceinline__ float dist_lane(const float4* q, const float* rows, uint32_t stride, uint32_t id, int metric) {
    const float4* r = reinterpret_cast<const float4*>(rows + uint64_t(id) * stride);
    float s = 0.0f;
    for (uint32_t c = 0; 4u * c < stride; ++c) {
        const float4 a = q[c], b = __ldg(r + c);
        if (metric == HNSW_L2SQ) {
            const float x = a.x - b.x, y = a.y - b.y, z = a.z - b.z, w = a.w - b.w;
            s = fmaf(x, x, s);
            s = fmaf(y, y, s);
            s = fmaf(z, z, s);
            s = fmaf(w, w, s);
        } else {
            s = fmaf(a.x, b.x, s);
            s = fmaf(a.y, b.y, s);
            s = fmaf(a.z, b.z, s);
            s = fmaf(a.w, b.w, s);
        }
    }
    return metric == HNSW_L2SQ ? s : 1.0f - s;
}

// Alg. 1's descent and layer insertion on layers >= 1 for each new element in
// turn: greedy descent above the element's level, then on each of its layers
// SEARCH-LAYER with efConstruction, SELECT-NEIGHBORS for its list and the
// reverse links, shrunk with the same selection beyond Mmax; a new top level
// makes the element the enter point (as in Alg. 1).
//
// The elements follow one another (each may link to the one before it), so one
// block does them all and what counts is the length of an element's chain.
// The search is the single-list form: W sorted by key with an 'expanded' bit
// below the id, its unexpanded entries playing C (an element that left W can
// never be expanded: it lies beyond W's furthest when reached); an expansion's
// new neighbours are merged at once (taking them one at a time keeps W = the
// ef smallest of W and the ones taken, in any order).  W lies in shared memory
// and, E entries per thread, in registers.  An expansion is
//  * every warp by itself finds the first unexpanded entry, from `scan` on;
//  * its neighbours are scored, up to NB by a warp.  The entry after it is
//    expanded next unless a nearer one turns up, so that one's neighbours,
//    vectors and visited tags are requested before the scoring is waited for
//    (a tag read that early misses the neighbours of the expansion in between:
//    they are compared with);
//  * each warp that holds entries looks the new keys' places in W up by binary
//    search; from them follow how far its entries move and, in the first warp,
//    where the keys go, all into the other copy of W.
// That is one block barrier, two where something entered W.
// Reverse links are independent of one another (each changes one list and
// reads vectors): a warp each.  Measured, 1,000 elements into 20,000, of which 70
// go to a layer of 1,250 (efConstruction 200, 128 coordinates): the whole
// insertion call took 99 ms with one warp here, and takes 28.5.  It took 24.5
// with distances added in parts by a warp's lanes: 440 cycles less an expansion,
// but other sums, which near-ties show in the lists (dist_seq).  Rows of 200:
// 130 ms with one warp, 38.4 now.  What bounds it is an expansion's
// instructions, which follow one another (3,100 cycles: 600 to find the entry,
// 1,000 to score, 400 for the requests, 2,000 where keys are merged, which is
// every other time), not the reads.  Slower or the same: 8 warps with a team of
// 8 lanes per row, visited elements as a bitmap in shared memory, vectors read
// past L1.  Rows above 128 coordinates spill 40 to 280 bytes at 128 registers.
template <int DW, int E, int NB>
__global__ void __launch_bounds__(kUpThreads) insert_upper(const UpperArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    UpperSmem<E>& S = *reinterpret_cast<UpperSmem<E>*>(smem);
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const DevIndex& V = a.v;
    const float* rows = reinterpret_cast<const float*>(V.vec);
    const uint32_t stride = V.row_chunks * 4;
    const int Mmax = int(V.Mmax), efc = a.efc;
    uint32_t epoch = 0;
    uint32_t ep = uint32_t(a.state[0]);
    int L = a.state[1];
    int kb = 0;  // which of S.K and S.ids an expansion uses
    for (int i = t; i < 2 * kMaxOld; i += kUpThreads) (&S.K[0][0])[i] = ~0ull;  // stay so from Mmax on
    for (uint32_t u = 0; u < a.n; ++u) {
        const uint32_t q = a.ids[u];
        const int l = a.lv[u];
        float4* const wt = S.t[wid];
        uint64_t cur;
        {  // the enter point's distance, added as the selection adds
            TeamVec<DW> x, y;
            load_team(rows, stride, q, x, lane);
            load_team(rows, stride, ep, y, lane);
            cur = mkkey(dist_team(x, y, V.metric, lane), ep);
        }
        __syncthreads();  // the last element's lists are written, its shared memory is read
        for (uint32_t c = t; 4u * c < stride; c += kUpThreads)
            S.q[c] = __ldg(reinterpret_cast<const float4*>(rows + uint64_t(q) * stride) + c);
        __syncthreads();
        int buf = 0;
        for (int lc = L; lc > l; --lc) {  // descent above the level, ef = 1 (steepest descent)
            for (;;) {
                const uint32_t* row = upper_row(a, kid(cur), lc);
                uint64_t best = ~0ull;
                for (int j = wid; j < Mmax; j += kUpWarps) {
                    const uint32_t e = row[j];
                    if (e == kNone) break;  // valid ids come first
                    float4 v[DW / 4];
                    load_warp<DW>(v, rows, stride, e, lane);
                    const uint64_t k = mkkey(dist_seq<DW>(S.q, v, stride, V.metric, wt, lane), e);
                    best = k < best ? k : best;
                }
                if (lane == 0) S.best[buf][wid] = best;
                __syncthreads();
                best = S.best[buf][lane & (kUpWarps - 1)];
#pragma unroll
                for (int o = kUpWarps / 2; o > 0; o >>= 1) {
                    const uint64_t other = __shfl_xor_sync(kFull, best, o);
                    best = other < best ? other : best;
                }
                buf ^= 1;
                if (best >= cur) break;
                cur = best;
            }
        }
        int n_ep = 1;
        if (t == 0) S.Ek[0] = cur;
        __syncthreads();
        for (int lc = l < L ? l : L; lc >= 1; --lc) {
            // SEARCH-LAYER(q, ep, efc, lc)
            ++epoch;
            uint64_t w[E];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int i = e * kUpThreads + t;
                w[e] = ~0ull;
                if (i < n_ep) {  // n_ep <= efc (the previous layer's W)
                    const uint64_t k = S.Ek[i];
                    a.visited[kid(k)] = epoch;
                    w[e] = (k & 0xffffffff00000000ull) | (uint64_t(kid(k)) << 1);
                }
                S.T[0][i] = w[e];
            }
            int cw = 0;              // which of S.T is W
            int scan = 0;            // the entries before it are expanded
            uint32_t ahead = kNone;  // the element whose neighbours these are:
            uint32_t ne[NB], tag[NB];
            float4 nv[NB][DW / 4];
            auto request = [&](uint32_t c, uint32_t first_row) {
                ahead = c;
                const uint32_t* row = V.nbrU + (uint64_t(first_row) + uint32_t(lc - 1)) * V.sU;
#pragma unroll
                for (int k = 0; k < NB; ++k) ne[k] = wid + k * kUpWarps < Mmax ? row[wid + k * kUpWarps] : kNone;
#pragma unroll
                for (int k = 0; k < NB; ++k)
                    if (ne[k] != kNone) {
                        tag[k] = a.visited[ne[k]];
                        load_warp<DW>(nv[k], rows, stride, ne[k], lane);
                    }
            };
            __syncthreads();
            for (;; kb ^= 1) {
                const uint64_t* T = S.T[cw];
                // the first unexpanded entry, and the one after it
                int p = -1;
                uint32_t c = kNone, c2 = kNone;
                for (int s0 = scan; s0 < efc; s0 += 32) {
                    const uint32_t lo = s0 + lane < efc ? uint32_t(T[s0 + lane]) : 1u;
                    unsigned m = __ballot_sync(kFull, !(lo & 1u));
                    if (!m && p >= 0) break;  // one more window at most for the second
                    if (m && p < 0) {
                        const int at = __ffs(m) - 1;
                        p = s0 + at;
                        c = __shfl_sync(kFull, lo >> 1, at);
                        m &= m - 1;
                    }
                    if (!m) continue;
                    c2 = __shfl_sync(kFull, lo >> 1, __ffs(m) - 1);
                    break;
                }
                if (p < 0) break;  // every entry of W expanded (Alg. 2 stops)
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (e * kUpThreads + t == p) w[e] |= 1ull;
                // its neighbours
                const uint64_t thr = T[efc - 1] & ~1ull;  // W's furthest (all ones but one bit: not full)
                const uint32_t row2 = c2 != kNone ? V.upoff[c2] : 0u;
                const bool early = c == ahead;
                if (!early) request(c, V.upoff[c]);
                const uint32_t o0 = early && lane < Mmax ? S.ids[kb ^ 1][lane] : kNone;
                const uint32_t o1 = early && lane + 32 < Mmax ? S.ids[kb ^ 1][lane + 32] : kNone;
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    const int j = wid + k * kUpWarps;
                    if (j >= Mmax) break;
                    uint64_t key = ~0ull;
                    const uint32_t e = ne[k];
                    if (e != kNone && !__any_sync(kFull, tag[k] == epoch || o0 == e || o1 == e)) {
                        const float dq = dist_seq<DW>(S.q, nv[k], stride, V.metric, wt, lane);
                        const uint64_t ke = (uint64_t(f2ord(dq)) << 32) | (uint64_t(e) << 1);
                        if (ke < thr) key = ke;
                    }
                    if (lane == 0) {
                        S.K[kb][j] = key;
                        S.ids[kb][j] = e;
                        if (e != kNone) a.visited[e] = epoch;
                    }
                }
                if (c2 != kNone) request(c2, row2);
                __syncthreads();
                const uint64_t kn[2] = {S.K[kb][lane], Mmax > 32 ? S.K[kb][lane + 32] : ~0ull};
                const unsigned mk[2] = {__ballot_sync(kFull, kn[0] != ~0ull), __ballot_sync(kFull, kn[1] != ~0ull)};
                if (!(mk[0] | mk[1])) {
                    // entries before `scan` are not looked at until a merge
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (e * kUpThreads + t == p) S.T[cw][p] = w[e];
                    scan = p + 1;
                    continue;
                }
                uint64_t* T2 = S.T[cw ^ 1];
                if (wid * 32 < efc) {
                    int lb[2] = {0, 0}, rank[2] = {0, 0}, above[E];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (mk[h])  // entries of W below the key, four ways a step
                            for (int step = 1 << ((31 - __clz(efc)) & ~1); step > 0; step >>= 2) {
                                const int b = lb[h] - 1;
                                int up = 0;
#pragma unroll
                                for (int x = 1; x <= 3; ++x)
                                    up += b + x * step < efc && T[b + x * step] < kn[h];
                                lb[h] += up * step;
                            }
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (kn[h] == ~0ull) lb[h] = INT_MAX;  // an empty slot lies below no entry
#pragma unroll
                    for (int e = 0; e < E; ++e) above[e] = 0;  // new keys below each entry
#pragma unroll
                    for (int g = 0; g < NB; ++g) {  // 16 slots at a time: their reads overlap
                        if (!(mk[g / 2] >> (16 * (g & 1)) & 0xffffu)) continue;
#pragma unroll
                        for (int x = 0; x < 16; ++x) {
                            const uint64_t k = S.K[kb][16 * g + x];
                            const int l0 = __shfl_sync(kFull, lb[g / 2], 16 * (g & 1) + x);
#pragma unroll
                            for (int e = 0; e < E; ++e) above[e] += l0 <= e * kUpThreads + t;
                            rank[0] += k < kn[0];
                            if (NB > 2) rank[1] += k < kn[1];
                        }
                    }
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int i = e * kUpThreads + t;
                        if (i < efc && i + above[e] < efc) T2[i + above[e]] = w[e];
                    }
                    if (wid == 0) {
                        int first = INT_MAX;
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            if (kn[h] != ~0ull) {
                                const int i = lb[h] + rank[h];
                                if (i < efc) T2[i] = kn[h];
                                first = min(first, i);
                            }
                        first = int(__reduce_min_sync(kFull, uint32_t(first)));
                        if (lane == 0) S.first = first;
                    }
                }
                __syncthreads();
                cw ^= 1;
                scan = min(p + 1, S.first);
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int i = e * kUpThreads + t;
                    w[e] = i < efc ? T2[i] : ~0ull;
                }
            }
            // the result: the first efc entries, and enter points of the next layer
            int have = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int i = e * kUpThreads + t;
                const bool in = i < efc && w[e] != ~0ull;
                if (in) S.Ek[i] = (w[e] & 0xffffffff00000000ull) | lid(w[e]);
                have += __syncthreads_count(in);
            }
            n_ep = have;
            // neighbourhood(q) at lc: SELECT-NEIGHBORS(q, W, M)
            if (wid == 0) {
                const int nr = select_links<DW>(
                    rows, stride, V.metric,
                    [&](int i, uint32_t& id, float& dist) {
                        id = kid(S.Ek[i]);
                        dist = kdist(S.Ek[i]);
                    },
                    n_ep, a.M, a.heuristic != 0, a.keep_pruned != 0, S.sel[0], lane);
                uint32_t* rq = upper_row(a, q, lc);
                for (int j = lane; j < Mmax; j += 32) rq[j] = j < nr ? S.sel[0].Rid[j] : kNone;
                for (int j = lane; j < nr; j += 32) S.qR[j] = S.sel[0].Rid[j];
                if (lane == 0) S.nr = nr;
            }
            __syncthreads();
            // reverse links and their shrink, a warp each
            for (int x = wid; x < S.nr; x += kUpWarps) {
                const uint32_t r = S.qR[x];
                uint32_t* rr = upper_row(a, r, lc);
                int n0 = 0;
                for (int j = lane; j < Mmax; j += 32) n0 += rr[j] != kNone;
                n0 = __reduce_add_sync(kFull, n0);
                if (n0 < Mmax) {
                    if (lane == 0) rr[n0] = q;
                    continue;
                }
                // the members and q by their distance to r, a lane each
                uint64_t* keys = S.keys[wid];
                __syncwarp();
                for (uint32_t c = lane; 4u * c < stride; c += 32)
                    wt[c] = __ldg(reinterpret_cast<const float4*>(rows + uint64_t(r) * stride) + c);
                __syncwarp();
                for (int j = lane; j <= n0; j += 32) {
                    const uint32_t c2 = j < n0 ? rr[j] : q;
                    keys[j] = mkkey(dist_lane(wt, rows, stride, c2, V.metric), c2);
                }
                int n2 = 32;
                while (n2 < n0 + 1) n2 <<= 1;
                for (int j = n0 + 1 + lane; j < n2; j += 32) keys[j] = ~0ull;
                __syncwarp();
                sort_keys(keys, n2, lane);
                const int nr2 = select_links<DW>(
                    rows, stride, V.metric,
                    [&](int i, uint32_t& id, float& dist) {
                        id = kid(keys[i]);
                        dist = kdist(keys[i]);
                    },
                    n0 + 1, Mmax, a.heuristic != 0, a.keep_pruned != 0, S.sel[wid], lane);
                for (int j = lane; j < Mmax; j += 32) rr[j] = j < nr2 ? S.sel[wid].Rid[j] : kNone;
                __syncwarp();
            }
            __syncthreads();
        }
        if (l > L) {  // a new top level moves the enter point
            ep = q;
            L = l;
        }
    }
    if (t == 0) {
        a.state[0] = int(ep);
        a.state[1] = L;
    }
}

// the instance for lists of up to Mmax (<= kMaxOld)
template <int DW, int E>
auto upper_kernel(int Mmax) {
    return Mmax <= kUpWarps       ? insert_upper<DW, E, 1>
           : Mmax <= 2 * kUpWarps ? insert_upper<DW, E, 2>
                                  : insert_upper<DW, E, 4>;
}
static_assert(kMaxOld <= 4 * kUpWarps, "a warp scores up to 4 neighbours");

hnsw_status ins_fail(hnsw_status st, const std::string& m) { return fail(st, "hnsw_insert: " + m); }

}  // namespace

extern "C" hnsw_status hnsw_reserve(hnsw_index* ix, uint64_t capacity, void* stream) {
    if (!ix) return fail(HNSW_EINVAL, "hnsw_reserve: null index");
    std::lock_guard<std::mutex> lk(ix->insert_mu);
    const DevIndex D = dev_snapshot(ix);
    if (capacity < D.N || capacity >= (1ull << 31)) return fail(HNSW_EINVAL, "hnsw_reserve: capacity out of range");
    if (capacity <= ix->capacity && ix->v_nbr0[1 - ix->active]) return HNSW_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return fail(HNSW_ECUDA, std::string("hnsw_reserve: ") + cudaGetErrorString(e));
    const hnsw_index_info& I = ix->info;
    const uint64_t N = D.N;
    const uint32_t d_pad32 = D.row_chunks32 * 4;
    const uint64_t Mm1 = ix->build_M > 1 ? ix->build_M - 1 : 1;
    const uint64_t ucap = ix->upper_rows + (capacity - N) * 2 / Mm1 + 1024;
    const bool alias32 = ix->d_vec32 && ix->d_vec32 == ix->d_vec;
    std::vector<void*> fresh;
    auto get = [&](size_t bytes) -> void* {
        void* p = nullptr;
        if (e == cudaSuccess) e = cudaMalloc(&p, bytes ? bytes : 16);
        if (e == cudaSuccess) fresh.push_back(p);
        return p;
    };
    void* vec = get(capacity * I.row_bytes);
    void* scale = ix->d_scale ? get(capacity * 4) : nullptr;
    void* vec32 = ix->d_vec32 && !alias32 ? get(capacity * d_pad32 * 4ull) : nullptr;
    void* n0[2] = {get(capacity * D.s0 * 4ull), get(capacity * D.s0 * 4ull)};
    void* uo[2] = {get(capacity * 4), get(capacity * 4)};
    void* nu[2] = {get(ucap * D.sU * 4ull), get(ucap * D.sU * 4ull)};
    if (e != cudaSuccess) {
        cudaGetLastError();
        for (void* p : fresh) cudaFree(p);
        return fail(HNSW_ENOMEM, "hnsw_reserve: device memory");
    }
    auto cp = [&](void* dst, const void* src, size_t bytes) {
        if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, s);
    };
    auto ff = [&](void* dst, size_t bytes) {
        if (e == cudaSuccess && bytes) e = cudaMemsetAsync(dst, 0xFF, bytes, s);
    };
    cp(vec, ix->d_vec, N * I.row_bytes);
    if (scale) cp(scale, ix->d_scale, N * 4);
    if (vec32) cp(vec32, ix->d_vec32, N * d_pad32 * 4ull);
    for (int v = 0; v < 2; ++v) {
        ff(n0[v], capacity * D.s0 * 4ull);
        ff(uo[v], capacity * 4);
        ff(nu[v], ucap * D.sU * 4ull);
    }
    cp(n0[0], ix->dev.nbr0, N * D.s0 * 4ull);
    cp(uo[0], ix->dev.upoff, N * 4);
    cp(nu[0], ix->dev.nbrU, ix->upper_rows * D.sU * 4ull);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        for (void* p : fresh) cudaFree(p);
        return fail(HNSW_ECUDA, std::string("hnsw_reserve: copy: ") + cudaGetErrorString(e));
    }
    // release the old arrays (both adjacency versions)
    std::vector<void*> old = {ix->d_vec, ix->d_scale};
    if (ix->d_vec32 && !alias32) old.push_back(ix->d_vec32);
    for (int v = 0; v < 2; ++v)
        for (void* p : {ix->v_nbr0[v], ix->v_upoff[v], ix->v_nbrU[v]}) old.push_back(p);
    for (void* p : old)
        if (p) cudaFree(p);
    ix->d_vec = vec;
    ix->d_scale = scale;
    ix->d_vec32 = alias32 ? vec : vec32;
    for (int v = 0; v < 2; ++v) {
        ix->v_nbr0[v] = n0[v];
        ix->v_upoff[v] = uo[v];
        ix->v_nbrU[v] = nu[v];
    }
    ix->active = 0;
    ix->d_nbr0 = n0[0];
    ix->d_upoff = uo[0];
    ix->d_nbrU = nu[0];
    ix->capacity = capacity;
    ix->upper_capacity = ucap;
    {
        std::lock_guard<std::mutex> dl(ix->dev_mu);
        ix->dev.vec = static_cast<const uint4*>(vec);
        ix->dev.scale = static_cast<const float*>(scale);
        ix->dev.vec32 = static_cast<const uint4*>(ix->d_vec32);
        ix->dev.nbr0 = static_cast<const uint32_t*>(n0[0]);
        ix->dev.upoff = static_cast<const uint32_t*>(uo[0]);
        ix->dev.urows = uint32_t(ucap);
        ix->dev.nbrU = static_cast<const uint32_t*>(nu[0]);
    }
    std::lock_guard<std::mutex> il(ix->dev_mu);
    ix->info.device_bytes = capacity * I.row_bytes + (scale ? capacity * 4 : 0) + (vec32 ? capacity * d_pad32 * 4ull : 0) +
                            2 * (capacity * D.s0 * 4ull + capacity * 4 + ucap * D.sU * 4ull) + kWorkSlots * 4;
    return HNSW_OK;
}

extern "C" hnsw_status hnsw_insert(hnsw_index* ix, const float* data, uint64_t n, const double* level_u, void* stream) {
    if (!ix) return ins_fail(HNSW_EINVAL, "null index");
    if (n == 0) return HNSW_OK;
    if (!data || !level_u) return ins_fail(HNSW_EINVAL, "null data or level_u");
    std::lock_guard<std::mutex> lk(ix->insert_mu);
    DevIndex V = dev_snapshot(ix);
    const uint64_t N0 = V.N;
    if (!ix->v_nbr0[1 - ix->active]) return ins_fail(HNSW_EINVAL, "no capacity reserved (hnsw_reserve)");
    if (N0 + n > ix->capacity) return ins_fail(HNSW_EINVAL, "beyond the reserved capacity");
    if (V.storage != HNSW_F32 && !V.vec32)
        return ins_fail(HNSW_EINVAL, "needs the fp32 vectors (F32 storage or keep_fp32_for_rerank)");
    if (N0 == 0) return ins_fail(HNSW_EINVAL, "the index is empty (build its first elements with hnsw_build)");
    if (V.d > 32u * kMaxDW) return ins_fail(HNSW_EINVAL, "d above 256");
    const int efc = int(ix->build_efC), M = int(ix->build_M), Mmax = int(V.Mmax), Mmax0 = int(V.Mmax0);
    const int heur = (ix->build_flags & 1u) ? 1 : 0, keep = (ix->build_flags & 4u) ? 1 : 0;
    if ((ix->build_flags & 2u) != 0) return ins_fail(HNSW_EINVAL, "graphs built with extendCandidates");
    if (efc < 1 || efc > 1024) return ins_fail(HNSW_EINVAL, "efConstruction of the graph outside 1..1024");
    // a list's rows and a selection's places are Mmax and Mmax0 (<= kMaxOld)
    if (M < 1 || M > Mmax || M > Mmax0) return ins_fail(HNSW_EINVAL, "M of the graph outside 1..min(Mmax, Mmax0)");
    // levels (the level draw of Alg. 1) and the new upper rows, in id order
    std::vector<uint8_t> lv(n);
    std::vector<uint32_t> up(n, kNone), U, Z;
    std::vector<uint8_t> Ul;
    uint64_t rows = ix->upper_rows;
    for (uint64_t i = 0; i < n; ++i) {
        const double u = level_u[i];
        if (!(u > 0.0 && u <= 1.0)) return ins_fail(HNSW_EINVAL, "level_u outside (0,1]");
        const double l = std::floor(-std::log(u) * ix->build_mL);
        if (l > 255) return ins_fail(HNSW_EINVAL, "level above 255");
        lv[i] = uint8_t(l);
        if (lv[i] > 0) {
            up[i] = uint32_t(rows);
            rows += lv[i];
            U.push_back(uint32_t(N0 + i));
            Ul.push_back(lv[i]);
        } else {
            Z.push_back(uint32_t(N0 + i));
        }
    }
    if (rows > ix->upper_capacity) return ins_fail(HNSW_EINVAL, "upper-layer rows beyond the reserved capacity");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // searches still reading the version about to be overwritten finish first
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return ins_fail(HNSW_ECUDA, cudaGetErrorString(e));
    const int act = ix->active, ina = 1 - act;
    const uint32_t d = V.d, d_pad32 = V.row_chunks32 * 4;
    DevBuf stage, dU, dUl, visited, state;
    auto alloc = [&](DevBuf& x, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(&x.p, bytes ? bytes : 16);
    };
    alloc(stage, n * d_pad32 * 4ull);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return ins_fail(HNSW_ENOMEM, "staging");
    }
    auto step = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
    };
    // the version to write: a copy of the published one, with the new rows empty
    step(cudaMemcpyAsync(ix->v_nbr0[ina], ix->v_nbr0[act], N0 * V.s0 * 4ull, cudaMemcpyDeviceToDevice, s));
    step(cudaMemcpyAsync(ix->v_upoff[ina], ix->v_upoff[act], N0 * 4, cudaMemcpyDeviceToDevice, s));
    step(cudaMemcpyAsync(ix->v_nbrU[ina], ix->v_nbrU[act], ix->upper_rows * V.sU * 4ull, cudaMemcpyDeviceToDevice, s));
    step(cudaMemsetAsync(static_cast<uint32_t*>(ix->v_nbr0[ina]) + N0 * V.s0, 0xFF, n * V.s0 * 4ull, s));
    step(cudaMemsetAsync(static_cast<uint32_t*>(ix->v_nbrU[ina]) + ix->upper_rows * V.sU, 0xFF,
                         (rows - ix->upper_rows) * V.sU * 4ull, s));
    step(cudaMemcpyAsync(static_cast<uint32_t*>(ix->v_upoff[ina]) + N0, up.data(), n * 4, cudaMemcpyHostToDevice, s));
    // the vectors: fp32 rows d_pad32 apart, then the stored form
    step(cudaMemsetAsync(stage.p, 0, n * d_pad32 * 4ull, s));
    step(cudaMemcpy2DAsync(stage.p, d_pad32 * 4ull, data, d * 4ull, d * 4ull, n, cudaMemcpyDefault, s));
    if (e != cudaSuccess) return ins_fail(HNSW_ECUDA, std::string("copy: ") + cudaGetErrorString(e));
    hnsw_status st = store_rows(ix, static_cast<const float*>(stage.p), N0, n, s);
    if (st != HNSW_OK) return st;
    // the fp32 view of the version being written
    V.nbr0 = static_cast<const uint32_t*>(ix->v_nbr0[ina]);
    V.upoff = static_cast<const uint32_t*>(ix->v_upoff[ina]);
    V.nbrU = static_cast<const uint32_t*>(ix->v_nbrU[ina]);
    V.urows = uint32_t(ix->upper_capacity);
    V.N = uint32_t(N0 + n);
    if (V.storage != HNSW_F32) {
        V.vec = V.vec32;
        V.row_chunks = V.row_chunks32;
        V.storage = HNSW_F32;
        V.scale = nullptr;
    }
    const int metric = V.metric;
    // 1. layer 0 of the new elements of level >= 1 (through the old upper layers)
    st = insert_layer0(ix, V, U, N0, metric, M, Mmax0, efc, heur, keep, s);
    if (st != HNSW_OK) return st;
    // 2. their upper layers, one at a time in id order
    if (!U.empty()) {
        alloc(dU, U.size() * 4);
        alloc(dUl, U.size());
        alloc(visited, (N0 + n) * 4);
        alloc(state, 16);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return ins_fail(HNSW_ENOMEM, "upper-layer buffers");
        }
        const int st0[2] = {int(V.ep), V.maxlevel};
        step(cudaMemcpyAsync(dU.p, U.data(), U.size() * 4, cudaMemcpyHostToDevice, s));
        step(cudaMemcpyAsync(dUl.p, Ul.data(), U.size(), cudaMemcpyHostToDevice, s));
        step(cudaMemsetAsync(visited.p, 0, (N0 + n) * 4, s));
        step(cudaMemcpyAsync(state.p, st0, 8, cudaMemcpyHostToDevice, s));
        UpperArgs ua{};
        ua.v = V;
        ua.ids = static_cast<const uint32_t*>(dU.p);
        ua.lv = static_cast<const uint8_t*>(dUl.p);
        ua.n = uint32_t(U.size());
        ua.efc = efc;
        ua.M = M;
        ua.Mmax = Mmax;
        ua.heuristic = heur;
        ua.keep_pruned = keep;
        ua.visited = static_cast<uint32_t*>(visited.p);
        ua.state = static_cast<int*>(state.p);
        const bool wide = V.row_chunks * 4 > 128, two = efc > kUpThreads;
        void (*up)(const UpperArgs) = wide ? (two ? upper_kernel<8, 2>(Mmax) : upper_kernel<8, 1>(Mmax))
                                           : (two ? upper_kernel<4, 2>(Mmax) : upper_kernel<4, 1>(Mmax));
        const size_t sm = two ? sizeof(UpperSmem<2>) : sizeof(UpperSmem<1>);
        {
            const hnsw_status r = raise_smem_limit(reinterpret_cast<const void*>(up), sm, "hnsw_insert");
            if (r != HNSW_OK) return r;
        }
        if (e == cudaSuccess) {
            up<<<1, kUpThreads, sm, s>>>(ua);
            e = cudaGetLastError();
        }
        int st1[2] = {0, 0};
        step(cudaMemcpyAsync(st1, state.p, 8, cudaMemcpyDeviceToHost, s));
        step(cudaStreamSynchronize(s));
        if (e != cudaSuccess) return ins_fail(HNSW_ECUDA, std::string("upper layers: ") + cudaGetErrorString(e));
        V.ep = uint32_t(st1[0]);
        V.maxlevel = st1[1];
    }
    // 3. layer 0 of the new elements of level 0
    st = insert_layer0(ix, V, Z, N0 + U.size(), metric, M, Mmax0, efc, heur, keep, s);
    if (st != HNSW_OK) return st;
    step(cudaStreamSynchronize(s));
    if (e != cudaSuccess) return ins_fail(HNSW_ECUDA, cudaGetErrorString(e));
    // publish the new version
    {  // the device view and the info together (both read under dev_mu)
        std::lock_guard<std::mutex> dl(ix->dev_mu);
        ix->dev.nbr0 = V.nbr0;
        ix->dev.upoff = V.upoff;
        ix->dev.nbrU = V.nbrU;
        ix->dev.urows = V.urows;
        ix->dev.N = V.N;
        ix->dev.ep = V.ep;
        ix->dev.maxlevel = V.maxlevel;
        ix->info.N = V.N;
        ix->info.max_level = V.maxlevel;
        ix->info.enter_point = V.ep;
        ix->info.n_upper_rows = rows;
    }
    ix->active = ina;
    ix->d_nbr0 = ix->v_nbr0[ina];
    ix->d_upoff = ix->v_upoff[ina];
    ix->d_nbrU = ix->v_nbrU[ina];
    ix->upper_rows = rows;
    ix->levels.insert(ix->levels.end(), lv.begin(), lv.end());
    return HNSW_OK;
}

extern "C" hnsw_status hnsw_index_to_blob(hnsw_index* ix, void** out_blob, uint64_t* out_bytes) {
    if (!ix || !out_blob || !out_bytes) return fail(HNSW_EINVAL, "hnsw_index_to_blob: null argument");
    std::lock_guard<std::mutex> lk(ix->insert_mu);
    const DevIndex D = dev_snapshot(ix);
    if (D.storage != HNSW_F32 && !D.vec32)
        return fail(HNSW_EINVAL, "hnsw_index_to_blob: needs the fp32 vectors (F32 storage or keep_fp32_for_rerank)");
    const uint64_t N = D.N;
    const uint32_t d = D.d, d_pad32 = D.row_chunks32 * 4;
    const BlobLayout lay = BlobLayout::of(N, d, D.Mmax0, D.Mmax, ix->upper_rows);
    uint8_t* b = static_cast<uint8_t*>(std::calloc(lay.total, 1));
    if (!b) return fail(HNSW_ENOMEM, "hnsw_index_to_blob: host memory");
    const void* src32 = D.storage == HNSW_F32 ? static_cast<const void*>(D.vec) : static_cast<const void*>(D.vec32);
    cudaError_t e = cudaMemcpy2D(b + lay.data, d * 4ull, src32, d_pad32 * 4ull, d * 4ull, N, cudaMemcpyDeviceToHost);
    std::vector<uint32_t> h0(N * size_t(D.s0)), hu(ix->upper_rows * size_t(D.sU));
    if (e == cudaSuccess && !h0.empty()) e = cudaMemcpy(h0.data(), D.nbr0, h0.size() * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && !hu.empty()) e = cudaMemcpy(hu.data(), D.nbrU, hu.size() * 4, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        std::free(b);
        return fail(HNSW_ECUDA, std::string("hnsw_index_to_blob: ") + cudaGetErrorString(e));
    }
    std::memcpy(b + lay.level, ix->levels.data(), N);
    for (uint64_t i = 0; i < N; ++i)
        for (uint32_t c = 0; c < D.Mmax0; ++c) wr<uint32_t>(b + lay.nbr0 + (i * D.Mmax0 + c) * 4, h0[i * D.s0 + c]);
    for (uint64_t r = 0; r < ix->upper_rows; ++r)
        for (uint32_t c = 0; c < D.Mmax; ++c) wr<uint32_t>(b + lay.nbrU + (r * D.Mmax + c) * 4, hu[r * D.sU + c]);
    BlobHeader h{};
    h.version = 1;
    h.metric = uint32_t(D.metric);
    h.N = N;
    h.d = d;
    h.M = ix->build_M;
    h.Mmax = D.Mmax;
    h.Mmax0 = D.Mmax0;
    h.maxlevel = N ? uint32_t(D.maxlevel) : 0;
    h.ep = N ? D.ep : kNone;
    h.flags = ix->build_flags;
    h.efC = ix->build_efC;
    h.mL = ix->build_mL;
    h.n_upper_rows = ix->upper_rows;
    h.checksum = checksum64(b + 128, lay.total - 128, nullptr);
    write_header(b, h);
    *out_blob = b;
    *out_bytes = lay.total;
    return HNSW_OK;
}
