// search_team.cuh -- K-NN-SEARCH with a block of warps per query, for batches
// that do not fill the GPU with a warp per query.
//
// Such a batch is bound by the latency of one query's chain of expansions
// (each: neighbour row, vector rows, merge), so the chain is taken apart:
//  * warp 0 keeps W and runs Alg. 2's sequence of expansions.  W is a sorted
//    list in its registers (entry i in lane i % 32); an expansion's new keys
//    are merged at once: every entry counts the new keys below it, every new
//    key the entries and new keys below it, and one pass through shared
//    memory puts all of them in place.
//  * every other warp holds a slot: an element of W whose neighbours it
//    scores ahead of the element's expansion.  After each expansion warp 0
//    gives free slots the first entries of W that have none; they are the
//    next to be expanded unless a nearer element is found meanwhile, and then
//    keep their slots until they are (or leave W).
// Warp 0 expands the first unexpanded entry of W as soon as its slot is
// ready: it takes the neighbours that are still unvisited and inserts them.
// The sequence of expansions and insertions is the warp-per-query kernel's,
// which is Alg. 2's; only the moment at which distances are computed differs.
// A slot's warp leaves out neighbours already in the visited set (they have
// been offered to W), and a neighbour visited between the scoring and the
// expansion is dropped at the expansion.
//
// Warp 0 and a slot's warp hand over by two named barriers per slot (command:
// warp 0 arrives, the slot's warp waits; ready: the other way round): hardware
// barriers inside one block, no polling.  Every command is followed by one
// wait for its result before the slot's next command.
//
// What bounds it: warp 0's own chain of dependent instructions (about 3,000
// cycles per expansion, of which select and slot assignment 600, visited test
// and waiting 1,200, merge 550); more slots than two per query change little.
// Measured (us per batch, warp per query / 8 warps / 4 warps): SIFT-shaped 1M,
// bf16 + rerank, ef 50: 1 query 131 / 96 / 98, 77: 304 / 237 / 248, 304: 358 /
// 272 / 301, 600: 363 / 409 / 311, 1,000: 400 / 577 / 456; GloVe-shaped 400k,
// fp32, k 100, ef 256: 1: 855 / 598 / 596, 304: 1,505 / 1,004 / 1,053, 600:
// 1,700 / 1,730 / 1,268, 1,000: 1,765 / 2,604 / 1,876.
#pragma once

#include "search_dev.cuh"

namespace hnswgb {

constexpr int kTeamMaxWarps = 8;       // warp 0 and up to 7 slots (2 named barriers each, ids 1..14)
constexpr uint32_t kTeamMaxN = 1u << 30;  // keys here keep two state bits below the id

// Control words of a block (off_ctl).
struct TeamCtl {
    uint64_t best[2][kTeamMaxWarps];  // descent: each warp's best neighbour (two steps' worth)
    uint32_t uoff[2][kTeamMaxWarps];  // and its first upper row
    uint32_t cnt[2][kTeamMaxWarps];   // and how many it scored
    uint32_t slot_el[kTeamMaxWarps];  // commands: element to score (kNone: the query is done)
    int size;                         // |W| at the end
    uint32_t next;
};

__device__ __forceinline__ void bar_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// true when id is in its home bucket of the visited set (an id that was
// displaced to another bucket is not found: its distance is computed again)
__device__ __forceinline__ bool visited(const uint32_t* H, int hlog, uint32_t id) {
    const uint4 v = reinterpret_cast<const uint4*>(H)[(id * 2654435761u) >> (34 - hlog)];
    return v.x == id || v.y == id || v.z == id || v.w == id;
}

// Inserts each lane's id (want: this lane has one; ids distinct) into the
// visited set; returns true where it was not there.  A full bucket sends the
// id to the next one, and a lane that lost a slot to another lane tries again,
// so the set forgets nothing until 8 buckets in a row are full; lossy is then
// set (in the lane that overwrote a slot).
__device__ __forceinline__ bool visit_all(uint32_t* H, int hlog, uint32_t id, bool want, bool& lossy) {
    const uint32_t mask = (1u << (hlog - 2)) - 1u;
    uint32_t b = (id * 2654435761u) >> (34 - hlog);
    bool pending = want, fresh = false;
    int probes = 0;
    do {
        uint32_t* at = nullptr;
        if (pending) {
            uint32_t* sl = H + 4 * b;
            const uint4 v = *reinterpret_cast<const uint4*>(sl);
            if (v.x == id || v.y == id || v.z == id || v.w == id) {
                pending = false;
            } else {
                const int slot = v.x == kNone ? 0 : (v.y == kNone ? 1 : (v.z == kNone ? 2 : (v.w == kNone ? 3 : -1)));
                if (slot >= 0) {
                    at = sl + slot;
                } else if (++probes < 8) {
                    b = (b + 1u) & mask;
                } else {
                    sl[id & 3u] = id;
                    lossy = true;
                    fresh = true;
                    pending = false;
                }
            }
        }
        __syncwarp();  // every lane has read its bucket before any writes into it
        if (at) *at = id;
        __syncwarp();
        if (at && *at == id) {
            fresh = true;
            pending = false;
        }
    } while (__any_sync(kFull, pending));
    return fresh;
}

// W of a query in the registers of one warp: lane l holds entries l, l + 32,
// ..., ascending.  key = ord(dist) << 32 | id << 2 | state; state 0: no slot,
// 1: has a slot, 3: expanded; an empty entry is all ones.  Entries from ef' on
// are ones that left W: never expanded, never returned.
template <int R>
struct RegList {
    uint64_t w[R];
    int r0;  // no unexpanded entry lies in the rows of 32 before this one

    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = ~0ull;
        r0 = 0;
    }
    // The first of the first ef entries that is not expanded (ke, at index
    // ie) and the first that has no slot either (ka, ia); all ones: none.
    __device__ __forceinline__ void find(int ef, uint64_t& ke, int& ie, uint64_t& ka, int& ia, int lane) {
        ke = ka = ~0ull;
        ie = ia = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r < r0 || (ke != ~0ull && ka != ~0ull)) continue;
            const bool in = r * 32 + lane < ef;
            const unsigned me = __ballot_sync(kFull, in && !(uint32_t(w[r]) & 2u));
            const unsigned ma = __ballot_sync(kFull, in && !(uint32_t(w[r]) & 3u));
            if (ke == ~0ull && me) {
                ie = r * 32 + __ffs(me) - 1;
                ke = __shfl_sync(kFull, w[r], ie);
                r0 = r;
            }
            if (ka == ~0ull && ma) {
                ia = r * 32 + __ffs(ma) - 1;
                ka = __shfl_sync(kFull, w[r], ia);
            }
        }
    }
    __device__ __forceinline__ void mark(int i, uint32_t bits, int lane) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r * 32 + lane == i) w[r] |= bits;
    }
    // state 0 for the entry with key k
    __device__ __forceinline__ void unmark(uint64_t k) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (w[r] == k) w[r] = k & ~3ull;
    }
    __device__ __forceinline__ bool has(uint64_t k) const {  // on some lane: an entry of k's element
        bool h = false;
#pragma unroll
        for (int r = 0; r < R; ++r) h |= (uint32_t(w[r]) | 3u) == (uint32_t(k) | 3u) && w[r] != ~0ull;
        return h;
    }
    // Merges the m (1..32) distinct keys K[0..m) (shared memory) into the
    // list; T: 32 R keys of shared memory, which then holds the list.
    __device__ __forceinline__ void merge(const uint64_t* K, int m, uint64_t* T, int lane) {
        const uint64_t mine = lane < m ? K[lane] : ~0ull;
        int c[R];  // new keys below each entry
#pragma unroll
        for (int r = 0; r < R; ++r) c[r] = 0;
        int pos = 0;  // entries and new keys below this lane's new key
        for (int j = 0; j < m; ++j) {
            const uint64_t k = K[j];
            pos += k < mine;
            int below = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool p = k < w[r];
                c[r] += p;
                below += 32 - __popc(__ballot_sync(kFull, p));
            }
            if (lane == j) pos += below;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = r * 32 + lane + c[r];
            if (i < 32 * R) T[i] = w[r];
        }
        if (lane < m && pos < 32 * R) T[pos] = mine;
        __syncwarp();
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = T[r * 32 + lane];
        if (R > 2) r0 = min(r0, int(__reduce_min_sync(kFull, lane < m ? uint32_t(pos) : 0xffffffffu)) >> 5);
        else r0 = 0;
    }
};

template <int ST, int TEAM, int CPL, int U, int R>
__global__ void __launch_bounds__(32 * kTeamMaxWarps, 2) hnsw_team_kernel(const SearchArgs a) {
    using D = Dist<ST, TEAM, CPL, U, false>;
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint64_t* W = reinterpret_cast<uint64_t*>(smem + a.off_vis);  // results only: in the visited set's bytes
    uint32_t* H = reinterpret_cast<uint32_t*>(smem + a.off_vis);
    TeamCtl& ctl = *reinterpret_cast<TeamCtl*>(smem + a.off_ctl);
    const DevIndex& ix = a.ix;
    const int deg = int(ix.Mmax0), slots = (max(deg, int(ix.Mmax)) + 31) & ~31;
    // this warp's slot: neighbour ids and their distances
    uint32_t* ids = reinterpret_cast<uint32_t*>(smem + a.off_slot) + w * 2 * slots;
    float* dst = reinterpret_cast<float*>(ids + slots);
    const int hsz = 1 << a.hlog;
    for (uint32_t qi = blockIdx.x; qi < a.n;) {
        int efq = a.efp, kq = a.k;
        uint64_t obase = uint64_t(qi) * uint64_t(a.k);
        if (a.q_kef) {
            const uint32_t v = __ldg(a.q_kef + qi);
            kq = int(v & 0xffffu);
            efq = max(kq, int(v >> 16));
            obase = __ldg(a.q_out + qi);
        }
        const float* qp = a.q + uint64_t(qi) * ix.d;
        float qr[D::QF];
        D::load_q(qp, ix.d, qr, lane);
        for (int i = threadIdx.x; i < (hsz >> 2); i += blockDim.x)
            reinterpret_cast<uint4*>(H)[i] = make_uint4(kNone, kNone, kNone, kNone);
        uint32_t n_eval = 0, n_exp0 = 0, n_stepU = 0;
        bool lossy = false;
        int size = 0;
        if (ix.N > 0) {
            // enter point and greedy descent (Alg. 5), the state in every
            // warp: a step's neighbours are split over the warps, each
            // warp's best (with its first upper row, read beside the
            // vectors) is exchanged through shared memory
            if (lane == 0) ids[0] = ix.ep;
            __syncwarp();
            D::run(ix, qr, ids, 1, dst, lane);
            __syncwarp();
            uint64_t cur = mkkey(dst[0], ix.ep);
            __syncwarp();
            n_eval = 1;
            uint32_t cur_uo = ix.maxlevel >= 1 ? __ldg(ix.upoff + ix.ep) : kNone;
            const int per = (int(ix.Mmax) + nw - 1) / nw;  // <= 32: at least 2 warps
            int buf = 0;
            for (int lc = ix.maxlevel; lc >= 1; --lc) {
                for (;;) {
                    const uint32_t* urow = ix.nbrU + (uint64_t(cur_uo) + uint64_t(lc - 1)) * ix.sU;
                    const int j = w * per + lane;
                    const uint32_t e = lane < per && j < int(ix.Mmax) ? __ldg(urow + j) : kNone;
                    const uint32_t uo = e != kNone ? __ldg(ix.upoff + e) : kNone;
                    const int n = __popc(__ballot_sync(kFull, e != kNone));  // valid ids come first
                    if (e != kNone) ids[lane] = e;
                    __syncwarp();
                    D::run(ix, qr, ids, n, dst, lane);
                    __syncwarp();
                    const uint64_t k = lane < n ? mkkey(dst[lane], e) : ~0ull;
                    const uint64_t kb = warp_min_u64(k);
                    if (lane < n ? k == kb : (n == 0 && lane == 0)) {
                        ctl.best[buf][w] = kb;
                        ctl.uoff[buf][w] = uo;
                        ctl.cnt[buf][w] = uint32_t(n);
                    }
                    __syncthreads();
                    const uint64_t v = lane < nw ? ctl.best[buf][lane] : ~0ull;
                    const uint64_t m = warp_min_u64(v);
                    n_eval += __reduce_add_sync(kFull, lane < nw ? ctl.cnt[buf][lane] : 0u);
                    ++n_stepU;  // one upper-layer element expanded (its row read)
                    const int at = __ffs(__ballot_sync(kFull, lane < nw && v == m)) - 1;
                    const uint32_t muo = ctl.uoff[buf][at];
                    buf ^= 1;
                    if ((m >> 1) >= (cur >> 1)) break;
                    cur = m;
                    cur_uo = muo;
                }
            }
            // layer 0 beam (Alg. 2 with ef')
            __syncthreads();  // the visited set is clear, the descent's exchanges are read
            if (w > 0) {
                // a slot: score the neighbours of the elements that warp 0 names
                for (;;) {
                    bar_sync(w);
                    const uint32_t c = ctl.slot_el[w];
                    if (c == kNone) break;
                    const uint32_t* nrow = ix.nbr0 + uint64_t(c) * ix.s0;
                    int n = 0;
                    for (int h = 0; h < deg; h += 32) {
                        const uint32_t e = h + lane < deg ? __ldg(nrow + h + lane) : kNone;
                        const bool add = e != kNone && !visited(H, a.hlog, e);
                        const unsigned m = __ballot_sync(kFull, add);
                        if (add) ids[n + __popc(m & lanemask_lt())] = e;
                        n += __popc(m);
                    }
                    for (int i = n + lane; i < slots; i += 32) ids[i] = kNone;
                    __syncwarp();
                    D::run(ix, qr, ids, n, dst, lane);
                    __syncwarp();
                    bar_arrive(kTeamMaxWarps - 1 + w);
                }
            } else {
                RegList<R> L;
                L.clear();
                if (lane == 0) L.w[0] = (cur & 0xffffffff00000000ull) | (uint64_t(key_id(cur)) << 2);
                visit_all(H, a.hlog, key_id(cur), lane == 0, lossy);
                uint64_t* K = reinterpret_cast<uint64_t*>(smem + a.off_merge);  // new keys of an expansion
                uint64_t* T = K + 32;                                            // W during a merge
                const unsigned all = (1u << nw) - 2u;  // the slots: warps 1 .. nw-1
                unsigned occ = 0u, busy = 0u;  // slots that hold an element; that are computing or not waited for yet
                uint64_t my_key = ~0ull;       // lane s: the element of slot s (state bits clear)
                uint64_t thr = ~0ull;          // the furthest entry of a full W (state bits clear)
                auto wait_slot = [&](int s) {
                    __syncwarp();
                    bar_sync(kTeamMaxWarps - 1 + s);
                    busy &= ~(1u << s);
                };
                auto give = [&](int s, uint64_t k) {  // element k (state bits clear) to slot s
                    if (busy >> s & 1u) wait_slot(s);
                    if (lane == s) my_key = k;
                    if (lane == 0) ctl.slot_el[s] = (uint32_t(k) >> 2);
                    __syncwarp();
                    bar_arrive(s);
                    occ |= 1u << s;
                    busy |= 1u << s;
                };
                for (;;) {
                    // free the slots of elements that left W, then give free
                    // slots the first entries that have none
                    occ &= ~__ballot_sync(kFull, my_key > thr && my_key != ~0ull);
                    uint64_t c, k;
                    int ic, ik;
                    L.find(efq, c, ic, k, ik, lane);
                    if (c == ~0ull) break;  // every entry of W expanded: Alg. 2 stops
                    while (k != ~0ull && occ != all) {
                        L.mark(ik, 1u, lane);
                        give(__ffs(all & ~occ) - 1, k);
                        if (occ == all) break;
                        L.find(efq, c, ic, k, ik, lane);
                    }
                    const uint64_t ck = c & ~3ull;
                    const bool in = occ >> lane & 1u;
                    unsigned at = __ballot_sync(kFull, in && my_key == ck);
                    if (!at) {
                        // all slots hold elements of W, none of them c: take the
                        // slot of the furthest one
                        const uint64_t far = ~warp_min_u64(in ? ~my_key : ~0ull);
                        at = __ballot_sync(kFull, in && my_key == far);
                        L.unmark(far | 1u);
                        L.mark(ic, 1u, lane);
                        give(__ffs(at) - 1, ck);
                    }
                    const int s = __ffs(at) - 1;
                    if (busy >> s & 1u) wait_slot(s);
                    L.mark(ic, 3u, lane);
                    occ &= ~(1u << s);
                    ++n_exp0;
                    const uint32_t* sid = reinterpret_cast<const uint32_t*>(smem + a.off_slot) + s * 2 * slots;
                    const float* sd = reinterpret_cast<const float*>(sid + slots);
                    for (int h = 0; h < deg; h += 32) {
                        const uint32_t e = sid[h + lane];
                        const float dd = sd[h + lane];
                        const bool fresh = visit_all(H, a.hlog, e, e != kNone, lossy);
                        n_eval += __popc(__ballot_sync(kFull, fresh));
                        const uint64_t key = (uint64_t(f2ord(dd)) << 32) | (uint64_t(e) << 2);
                        bool ok = fresh && key < thr;
                        unsigned mk = __ballot_sync(kFull, ok);
                        if (__any_sync(kFull, lossy)) {  // a forgotten element may still be in W
                            for (unsigned b = mk; b; b &= b - 1) {
                                const int l = __ffs(b) - 1;
                                if (__any_sync(kFull, L.has(__shfl_sync(kFull, key, l))) && lane == l) ok = false;
                            }
                            mk = __ballot_sync(kFull, ok);
                        }
                        if (!mk) continue;
                        // a new entry of W is likely to be expanded: its neighbour row into L2
                        if (ok) prefetch_l2(ix.nbr0 + uint64_t(e) * ix.s0);
                        if (ok) K[__popc(mk & lanemask_lt())] = key;
                        __syncwarp();
                        L.merge(K, __popc(mk), T, lane);
                        thr = T[efq - 1] & ~3ull;
                        if (thr == ~3ull) thr = ~0ull;  // W is not full
                        __syncwarp();
                    }
                }
                for (int s = 1; s < nw; ++s) {  // collect what is still computed, release the slots' warps
                    if (busy >> s & 1u) wait_slot(s);
                    if (lane == 0) ctl.slot_el[s] = kNone;
                    __syncwarp();
                    bar_arrive(s);
                }
                // W into shared memory, in the other kernels' key format
                int have = 0;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (r * 32 + lane < efq && L.w[r] != ~0ull) {
                        W[r * 32 + lane] = (L.w[r] & 0xffffffff00000000ull) | (uint64_t(uint32_t(L.w[r]) >> 2) << 1);
                        ++have;
                    }
                }
                have = __reduce_add_sync(kFull, have);
                lossy = __any_sync(kFull, lossy);
                if (lane == 0) ctl.size = have;
            }
            __syncthreads();
            size = ctl.size;
        }
        // results (the K nearest of W, Alg. 5)
        if (a.rerank && size > 0) {
            float* qs = reinterpret_cast<float*>(smem + a.off_qs);
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < ix.row_chunks32 * 4; i += blockDim.x) qs[i] = i < ix.d ? qp[i] : 0.0f;
            __syncthreads();
            dist32_rows(
                ix, qs, [&](int r) { return key_id(W[r]); }, 4 * w, 4 * nw, size,
                [&](int r, float v) { W[r] = mkkey(v, key_id(W[r])); }, lane);
            for (int i = size + threadIdx.x; i < a.efcap; i += blockDim.x) W[i] = ~0ull;
            __syncthreads();
            // keys are distinct: W needs no sort when every adjacent pair is in order
            bool unsorted = false;
            for (int i = threadIdx.x; i + 1 < size; i += blockDim.x) unsorted |= W[i] > W[i + 1];
            if (__syncthreads_or(unsorted)) {
                for (int kk = 2; kk <= a.efcap; kk <<= 1)  // bitonic sort
                    for (int j = kk >> 1; j > 0; j >>= 1) {
                        for (int i = threadIdx.x; i < a.efcap; i += blockDim.x) {
                            const int p = i ^ j;
                            if (p > i) {
                                const uint64_t x = W[i], y = W[p];
                                if ((x > y) == ((i & kk) == 0)) {
                                    W[i] = y;
                                    W[p] = x;
                                }
                            }
                        }
                        __syncthreads();
                    }
            }
        }
        for (int i = threadIdx.x; i < kq; i += blockDim.x) {
            const uint64_t kk = i < size ? W[i] : 0ull;
            a.out_ids[obase + i] = i < size ? key_id(kk) : kNone;
            a.out_dists[obase + i] = i < size ? key_dist(kk) : __int_as_float(0x7f800000);
        }
        if (a.stats && threadIdx.x == 0) {
            hnsw_query_stats s;
            s.n_eval = n_eval;
            s.n_exp0 = n_exp0;
            s.n_stepU = n_stepU;
            s.flags = lossy ? 1u : 0u;
            a.stats[qi] = s;
        }
        if (a.n <= gridDim.x) break;
        if (threadIdx.x == 0) ctl.next = gridDim.x + atomicAdd(a.work, 1u);
        __syncthreads();  // the next query's number; this query's W is read
        qi = ctl.next;
    }
}

}  // namespace hnswgb
