// search_kernel.cuh -- the one-warp-per-query search kernel (described in
// search.cu) and the choice of its instantiation; instantiated per storage
// type in search_f32.cu, search_bf16.cu, search_f16.cu and search_fp8.cu.
#pragma once

#include "search_dev.cuh"

namespace hnswgb {

// ---- deferred queries (mode 0) ----------------------------------------------
// Both run on one lane.  A claim takes the next ticket (one atomic, no
// retries) and waits for that slot's record -- written by a warp that holds
// the slot and is running -- or, when every query of the input queue has
// passed its decision and the slot was never pushed, gives up the ticket.
// The warps it waits for hold input-queue queries already (the queue is
// drained before any claim) and decide right after their descent.  The wait
// is bounded (2^20 polls, 0.1 to 1 s): a record that does not appear by then
// sets the error word and the claim gives up.
constexpr int kDeferSpin = 1 << 20;
constexpr uint32_t kDeferWarmup = 32;  // descents seen before any is deferred
// the automatic schedule defers in batches of up to 2^24 queries (256 MB of
// records); in larger ones the tail is a small part of the batch
constexpr uint64_t kDeferAutoMax = 1ull << 24;

__device__ __forceinline__ uint32_t ld_volatile_u32(const uint32_t* p) {
    return *reinterpret_cast<const volatile uint32_t*>(p);
}

// A pushed record (its .w = query index), or .w = kNone when none is left.
inline __device__ uint4 claim_deferred(const SearchArgs& a) {
    uint32_t* ctl = a.dfr_ctl;
    const uint32_t d = atomicAdd(ctl + 1, 1u);
    if (d >= a.n) return make_uint4(0u, 0u, 0u, kNone);
    const uint32_t* rw = reinterpret_cast<const uint32_t*>(a.dfr_rec + d);
    for (int it = 0; it < kDeferSpin; ++it) {
        const uint32_t q = ld_volatile_u32(rw + 3);
        if (q != kNone) {
            __threadfence();
            return make_uint4(ld_volatile_u32(rw), ld_volatile_u32(rw + 1), ld_volatile_u32(rw + 2), q);
        }
        if (ld_volatile_u32(ctl + 5) >= a.n) {  // every decision made: the pushes are final
            __threadfence();
            if (d >= ld_volatile_u32(ctl + 0)) return make_uint4(0u, 0u, 0u, kNone);
        }
        __nanosleep(128);
    }
    atomicExch(ctl + 2, 1u);
    if (a.err) {
        *reinterpret_cast<volatile uint32_t*>(a.err) = 1u;
        __threadfence_system();
    }
    return make_uint4(0u, 0u, 0u, kNone);
}

// Pushes query qi (layer-0 enter key, upper-layer counters) when its descent
// distance is below the mean of those seen before it; counts the decision
// (after the record is written) either way and returns whether it pushed.
inline __device__ bool maybe_defer(const SearchArgs& a, uint32_t qi, uint64_t cur, uint32_t n_eval, uint32_t n_stepU) {
    uint32_t* ctl = a.dfr_ctl;
    const float d1 = key_dist(cur);
    const uint32_t seen = atomicAdd(ctl + 3, 1u);
    const float sum = atomicAdd(reinterpret_cast<float*>(ctl + 4), d1);
    const bool push = seen >= kDeferWarmup && d1 * float(seen) < sum && n_eval < (1u << 20) && n_stepU < (1u << 12);
    if (push) {
        const uint32_t s = atomicAdd(ctl + 0, 1u);
        volatile uint32_t* rw = reinterpret_cast<volatile uint32_t*>(a.dfr_rec + s);
        rw[0] = uint32_t(cur);
        rw[1] = uint32_t(cur >> 32);
        rw[2] = (n_stepU << 20) | n_eval;
        __threadfence();
        rw[3] = qi;
    }
    __threadfence();
    if (!(a.dfr_hold && qi == 0)) atomicAdd(ctl + 5, 1u);
    return push;
}

// ---- the kernel -------------------------------------------------------------
// STOP: the build with learned-stop checks and trace recording (the plain
// search is compiled without them and keeps its smaller register budget).
// One learned-stop check of a warp's search: the six features of the state
// of W (aux: 1/d1, log1p(d1), layer-0 distance evaluations at entry) written
// to aux[4..9], and the network's logit (0 without a network).  log1p of the
// per-check features is taken as log(1 + x) with the fast logarithm.
HNSW_STOP_FN float stop_check(const StopDev* model, const uint64_t* W, int size, int kq, float* aux,
                              uint32_t n_eval0, uint32_t stale, float* hs, int lane) {
    const float inv_d1 = aux[0];
    float f[kStopIn];
    f[0] = __logf(1.0f + fmaxf(key_dist(W[0]) * inv_d1, 0.0f));
    f[1] = __logf(1.0f + fmaxf(key_dist(W[size - 1]) * inv_d1, 0.0f));
    f[2] = __logf(1.0f + float(n_eval0));
    f[3] = aux[1];
    f[4] = __logf(1.0f + float(stale));
    f[5] = __logf(1.0f + fmaxf(key_dist(W[kq - 1]) * inv_d1, 0.0f));
    float fv = f[0];
#pragma unroll
    for (int i = 1; i < kStopIn; ++i) fv = lane == i ? f[i] : fv;
    if (lane < kStopIn) aux[4 + lane] = fv;
    return model ? stop_logit<true>(model, f, hs, lane) : 0.0f;
}

// Register budget of each instantiation (per thread): 56 -- 9 blocks of 128
// threads resident per SM, 36 warps -- for the 2-lane teams of low-d rows, but
// for narrow searches with the stop on rows of one chunk, which spill 52 to 80
// bytes at 56 (8 bf16 coordinates, 10,000 queries at ef 50: 329 us at 56, 285
// at 64); 72 for fp32 rows of 128 coordinates (80 with the stop, the bounds
// checks or partial rows); more for more rows in flight (fp8 with 8 rows per
// team, f16 with 4); 64 (8 blocks) otherwise.  Full bf16 rows at 56 registers
// spill 20 bytes and run slower in spite of 4 more warps (10,000 queries at ef
// 50: 543 us against 520; low-d rows at 64: 1,047 against 989).  Partial fp32
// rows spill 4 to 32 bytes at 80, and are quicker so than with fewer warps: 100
// coordinates, 10,000 queries at ef 128, 717 us at 80, 805 at 88 without a
// spill (ef 50: the same).  Full fp32 rows with the stop and a wide W spill 8
// bytes there.  Without an explicit budget the compiler chose budgets that
// spilled.  Blocks of up to 256 threads are allowed so that large
// per-warp state (wide beams) can be packed into the shared memory of an SM
// (see the launch).
template <int ST, int TEAM, int CPL, int U, bool FULL, bool STOP, bool WIDE, bool CHECK>
constexpr int search_max_regs() {
    return (ST == HNSW_F32 && CPL == 4) ? ((STOP || CHECK || !FULL) ? 80 : 72)
         : (ST == HNSW_FP8E4M3 && U == 8) ? 96
         : (ST == HNSW_F16 && U == 4) ? 80
         : (TEAM == 2 && !CHECK && !(STOP && !FULL && !WIDE)) ? 56
                                 : 64;
}

// CHECK: the bounds-checked build (hnsw_search_params.check_bounds): every
// element id read from the graph is tested against N and every upper-row
// index against the rows allocated before any use; a query that meets a bad
// one sets stats flag bit 2 and leaves its search (its results are what W
// holds), with no device fault and no trap.
// WIDE: launches whose W may hold more than 64 entries, or whose layer-0
// lists more than 32 (merge_wide).
template <int ST, int TEAM, int CPL, int U, bool FULL, bool STOP, bool WIDE, bool CHECK = false>
__global__ void __launch_bounds__(256) __maxnreg__((search_max_regs<ST, TEAM, CPL, U, FULL, STOP, WIDE, CHECK>()))
    hnsw_search_kernel(const SearchArgs a) {
    using D = Dist<ST, TEAM, CPL, U, FULL>;
    // full fp32 rows of 128 coordinates have no registers left for the wide
    // merge's ballots at 72 (56 bytes of spill, 5% slower at ef 66 to 100)
    constexpr bool kBallot = search_max_regs<ST, TEAM, CPL, U, FULL, STOP, WIDE, CHECK>() != 72;
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & 31;
    uint8_t* wbase = smem + (threadIdx.x >> 5) * a.warp_smem;
    uint64_t* W = reinterpret_cast<uint64_t*>(wbase);
    uint32_t* H = reinterpret_cast<uint32_t*>(wbase + a.efcap * 8);
    uint32_t* ids = H + (1 << a.hlog);
    float* dst = reinterpret_cast<float*>(ids + kMaxNbr);
    uint32_t* nbuf = reinterpret_cast<uint32_t*>(dst + kMaxNbr);  // staged neighbour row (16-byte aligned)
    // per-query scalars read only at stop checks (kept out of registers):
    // 1/d1, log1p(d1), n_eval at layer 0 entry, checks recorded; [4..9] the
    // features of the last check
    float* aux = reinterpret_cast<float*>(nbuf + kMaxNbr);
    uint32_t* n_checks = reinterpret_cast<uint32_t*>(aux + 3);
    const DevIndex& ix = a.ix;
    const int hsz = 1 << a.hlog;
    for (;;) {
        uint32_t qi = 0;
        if (lane == 0) qi = atomicAdd(a.work, 1u);
        qi = __shfl_sync(kFull, qi, 0);
        // a deferred query taken up again (its enter key and counters parked
        // in aux words 10-12 until the beam starts)
        bool resumed = false;
        if (qi >= a.n) {
            if (CHECK || !a.dfr_ctl) break;
            // the input queue is drained: the deferred queries' beams
            if (lane == 0) {
                const uint4 r = claim_deferred(a);
                uint32_t* park = reinterpret_cast<uint32_t*>(aux) + 10;
                park[0] = r.x;
                park[1] = r.y;
                park[2] = r.z;
                qi = r.w;
            }
            qi = __shfl_sync(kFull, qi, 0);
            if (qi == kNone) break;
            resumed = true;
        }
        if (a.mode == 2) qi = __ldg(a.order + qi);
        const float* qp = a.q + uint64_t(qi) * ix.d;
        // per-query k and ef of a grouped launch (k is reread where needed so
        // that only ef stays live through the search)
        int efq = a.efp;
        if (a.q_kef) {
            const uint32_t v = __ldg(a.q_kef + qi);
            efq = max(int(v & 0xffffu), int(v >> 16));
        }
        float qr[D::QF];
        D::load_q(qp, ix.d, qr, lane);
        for (int i = lane; i < (hsz >> 2); i += 32)
            reinterpret_cast<uint4*>(H)[i] = make_uint4(kNone, kNone, kNone, kNone);
        uint32_t n_eval = 0, n_exp0 = 0, n_stepU = 0, flags = 0;
        if (STOP && lane == 0) *n_checks = 0;
        int size = 0;
        __syncwarp();
        bool bad = CHECK && ix.N > 0 && !(ix.ep < ix.N);  // bounds-checked build: a bad id or row met
        if (ix.N > 0 && !bad) {
            uint64_t cur = 0;
            if (resumed) {  // the descent ran before the query was deferred
                const uint32_t* park = reinterpret_cast<const uint32_t*>(aux) + 10;
                cur = (uint64_t(park[1]) << 32) | park[0];
                n_eval = park[2] & 0xfffffu;
                n_stepU = park[2] >> 20;
            } else if (a.mode == 2) {  // the descent ran in the first pass
                cur = a.ep_keys[qi];
                n_eval = a.up_cnt[2 * uint64_t(qi)];
                n_stepU = a.up_cnt[2 * uint64_t(qi) + 1];
            } else {
            // enter point and greedy descent (Alg. 5)
            if (lane == 0) ids[0] = ix.ep;
            __syncwarp();
            D::run(ix, qr, ids, 1, dst, lane);
            __syncwarp();
            cur = mkkey(dst[0], ix.ep);
            n_eval = 1;
            uint32_t cur_uo = ix.maxlevel >= 1 ? __ldg(ix.upoff + key_id(cur)) : kNone;  // cur's first upper row
            for (int lc = ix.maxlevel; lc >= 1 && !bad; --lc) {
                for (;;) {
                    const uint64_t row = uint64_t(cur_uo) + uint64_t(lc - 1);
                    if (CHECK && !(row < ix.urows)) {  // c absent from layer lc, or a bad offset
                        bad = true;
                        break;
                    }
                    const uint32_t* urow = ix.nbrU + row * ix.sU;
                    int n = 0;
                    __syncwarp();
                    for (int h = 0; h < int(ix.Mmax); h += 32) {
                        const int j = h + lane;
                        uint32_t e = j < int(ix.Mmax) ? __ldg(urow + j) : kNone;
                        if (CHECK && e != kNone && !(e < ix.N)) {
                            bad = true;
                            e = kNone;
                        }
                        const bool v = e != kNone;
                        const unsigned m = __ballot_sync(kFull, v);
                        if (v) ids[n + __popc(m & lanemask_lt())] = e;
                        n += __popc(m);
                    }
                    if (CHECK && __any_sync(kFull, bad)) {
                        bad = true;
                        break;
                    }
                    __syncwarp();
                    D::run(ix, qr, ids, n, dst, lane);
                    __syncwarp();
                    n_eval += n;
                    ++n_stepU;  // one upper-layer element expanded (its row read)
                    uint64_t kb = ~0ull;
                    for (int j = lane; j < n; j += 32) kb = min(kb, mkkey(dst[j], ids[j]));
                    kb = warp_min_u64(kb);
                    if ((kb >> 1) < (cur >> 1)) {
                        cur = kb;
                        cur_uo = __ldg(ix.upoff + key_id(kb));
                    } else {
                        break;
                    }
                }
            }
            }
            if (a.mode == 1) {  // first pass: keep the layer-0 enter point for the second
                if (lane == 0) {
                    a.ep_keys[qi] = cur;
                    a.up_cnt[2 * uint64_t(qi)] = n_eval;
                    a.up_cnt[2 * uint64_t(qi) + 1] = n_stepU;
                }
                __syncwarp();
                continue;
            }
            if (!CHECK && a.dfr_ctl && !resumed) {
                bool deferred = false;
                if (lane == 0) deferred = maybe_defer(a, qi, cur, n_eval, n_stepU);
                if (__shfl_sync(kFull, deferred, 0)) continue;  // its beam runs later
            }
            // layer 0 beam (Alg. 2 with ef')
            if (lane == 0) {
                W[0] = cur & ~1ull;
                visit_new(H, a.hlog, key_id(cur), flags);
            }
            size = 1;
            int scan = 0;
            const int deg = int(ix.Mmax0);
            if (STOP && lane == 0) {
                const float d1 = key_dist(cur);  // where the upper-layer descent ended
                aux[0] = 1.0f / fmaxf(d1, 1e-12f);
                aux[1] = log1pf(fmaxf(d1, 0.0f));
                aux[2] = __uint_as_float(n_eval);
            }
            // stale (expansions since the K nearest of W last changed) in the
            // high half, expansions left to the next check in the low half
            uint32_t stale_cd = STOP ? uint32_t(a.stop_period) : 0u;
            uint32_t nxt_id = kNone;  // element whose neighbour row is staged in nbuf
            __syncwarp();
            for (;;) {
                if (CHECK && bad) break;  // the descent met a bad id or row: W holds its last element
                int p = -1;
                // the window of W where p was found: its unexpanded entries
                // (bit per lane) and this lane's entry, for the next one after p
                unsigned win_m = 0u;
                uint32_t win_id = 0u;
                for (int s = scan; s < size; s += 32) {
                    // the low word of a key holds the id and the expanded bit
                    const int i = s + lane;
                    const uint32_t wlo = i < size ? reinterpret_cast<const uint32_t*>(W)[2 * i] : 1u;
                    const bool un = !(wlo & 1u);
                    const unsigned m = __ballot_sync(kFull, un);
                    if (m) {
                        const int b = __ffs(m) - 1;
                        p = s + b;
                        win_m = b < 31 ? (m & (~0u << (b + 1))) : 0u;
                        win_id = (wlo >> 1) & 0x7fffffffu;
                        break;
                    }
                }
                if (p < 0) {  // every entry of W expanded: Alg. 2 stops
                    if (nxt_id != kNone) cp_async_wait_all();
                    break;
                }
                const uint64_t kc = W[p];
                __syncwarp();
                if (lane == 0) W[p] = kc | 1ull;
                ++n_exp0;
                const uint32_t c = key_id(kc);
                const uint32_t* nrow = ix.nbr0 + uint64_t(c) * ix.s0;
                // was this row staged in shared memory during the previous expansion?
                const bool staged = c == nxt_id;
                if (nxt_id != kNone) {
                    cp_async_wait_all();
                    __syncwarp();
                }
                uint32_t e0 = kNone, e1 = kNone;
                if (staged) {
                    e0 = lane < deg ? nbuf[lane] : kNone;
                    if (WIDE && deg > 32) e1 = lane + 32 < deg ? nbuf[32 + lane] : kNone;
                } else {
                    e0 = lane < deg ? __ldg(nrow + lane) : kNone;
                    if (WIDE && deg > 32) e1 = lane + 32 < deg ? __ldg(nrow + 32 + lane) : kNone;
                }
                __syncwarp();
                if (CHECK && __any_sync(kFull, (e0 != kNone && !(e0 < ix.N)) || (e1 != kNone && !(e1 < ix.N)))) {
                    bad = true;  // no copy is in flight here: the staged row was waited for above
                    nxt_id = kNone;
                    break;
                }
#if HNSW_PREFETCH_NEXT
                // the next unexpanded entry after p is expanded next unless this
                // batch inserts a better element: stage its neighbour row now
                nxt_id = kNone;
                {
                    // within the window of p when it holds one, else the 32
                    // entries after p
                    unsigned m = win_m;
                    uint32_t id = win_id;
                    if (!m) {
                        const int i = p + 1 + lane;
                        const uint32_t wlo = i < size ? reinterpret_cast<const uint32_t*>(W)[2 * i] : 1u;
                        m = __ballot_sync(kFull, !(wlo & 1u));
                        id = (wlo >> 1) & 0x7fffffffu;
                    }
                    if (m) {
                        nxt_id = __shfl_sync(kFull, id, __ffs(m) - 1);
                        const uint32_t* np = ix.nbr0 + uint64_t(nxt_id) * ix.s0;
                        if (lane * 4 < deg) cp_async16(nbuf + lane * 4, np + lane * 4);
                        cp_async_commit();
                    }
                }
#endif
                int n = 0;
                {
                    const bool nw = e0 != kNone && visit_new(H, a.hlog, e0, flags);
                    const unsigned m = __ballot_sync(kFull, nw);
                    if (nw) ids[__popc(m & lanemask_lt())] = e0;
                    n = __popc(m);
                }
                if (WIDE && deg > 32) {
                    const bool nw = e1 != kNone && visit_new(H, a.hlog, e1, flags);
                    const unsigned m = __ballot_sync(kFull, nw);
                    if (nw) ids[n + __popc(m & lanemask_lt())] = e1;
                    n += __popc(m);
                }
                __syncwarp();
                int first_new = INT_MAX;
                if (n > 0) {
#if HNSW_PREFETCH_ROWS
                    // rows beyond the first gather round: start their DRAM reads now
                    if (n > D::RPR) {
                        for (int j = D::RPR + lane; j < n; j += 32) {
                            const uint8_t* rp =
                                reinterpret_cast<const uint8_t*>(ix.vec + uint64_t(ids[j]) * ix.row_chunks);
                            for (uint32_t b = 0; b < ix.row_chunks * 16; b += 128) prefetch_l2(rp + b);
                        }
                    }
#endif
                    D::run(ix, qr, ids, n, dst, lane);
                    __syncwarp();
                    n_eval += n;
                    for (int h = 0; h < (WIDE ? n : 1); h += 32) {
                        const int j = h + lane;
                        bool ok = j < n;
                        const uint64_t key = ok ? mkkey(dst[j], ids[j]) : 0ull;
                        first_new = min(first_new, WIDE && (CHECK || size > kNarrow)
                                                   ? merge_wide<kBallot>(W, size, efq, key, ok, lane)
                                                   : merge_small(W, size, efq, key, ok, lane));
                    }
                }
                scan = min(p + 1, first_new);
                if (STOP && a.stop_period > 0) {
                    const int kq = a.q_kef ? int(__ldg(a.q_kef + qi) & 0xffffu) : a.k;
                    // stale: expansions since an element entered the K nearest of W
                    // (once W holds K entries: since its K-th key last decreased),
                    // saturating at 65535
                    stale_cd = first_new < kq ? (stale_cd & 0xffffu) : __vaddus2(stale_cd, 0x10000u);
                    stale_cd -= 1u;
                    bool check = (stale_cd & 0xffffu) == 0u;
                    if (HNSW_STOP_SKIP_IMPROVING && check && !a.tr_count && first_new < kq) {
                        check = false;  // put off to the next expansion
                        stale_cd |= 1u;
                    }
                    if (check) stale_cd |= uint32_t(a.stop_period);
                    if (size >= kq && check) {
                        __syncwarp();
                        const StopDev* model = a.stop;  // global memory, read through L1
                        const float logit = stop_check(model, W, size, kq, aux, n_eval - __float_as_uint(aux[2]),
                                                       stale_cd >> 16, reinterpret_cast<float*>(wbase + a.off_hs), lane);
                        if (a.tr_count) {
                            __syncwarp();
                            const uint32_t c = *n_checks;
                            if (c < uint32_t(a.tr_max)) {
                                const uint64_t slot = uint64_t(qi) * uint64_t(a.tr_max) + c;
                                if (lane < kStopIn) a.tr_feat[slot * kStopIn + lane] = aux[4 + lane];
                                if (lane == 0 && a.tr_logit) a.tr_logit[slot] = logit;
                                for (int i = lane; i < a.k; i += 32) a.tr_topk[slot * uint64_t(a.k) + i] = key_id(W[i]);
                            }
                            __syncwarp();
                            if (lane == 0) *n_checks = c + 1;
                        } else if (model && logit > a.stop_logit) {
                            flags |= 2u;  // learned stop: W's top-K is predicted final
                            if (nxt_id != kNone) cp_async_wait_all();
                            __syncwarp();
                            break;
                        }
                    }
                }
            }
        }
        // results (the K nearest of W, Alg. 5)
        if (a.rerank && size > 0) {
            float* qs = reinterpret_cast<float*>(wbase + a.off_qs);
            const float* qrow = a.q + uint64_t(qi) * ix.d;  // re-derived: keeps qp out of the loop's registers
            __syncwarp();
            for (uint32_t i = lane; i < ix.row_chunks32 * 4; i += 32) qs[i] = i < ix.d ? qrow[i] : 0.0f;
            __syncwarp();
            for (int b = 0; b < size; b += kMaxNbr) {
                const int nb = min(kMaxNbr, size - b);
                for (int i = lane; i < nb; i += 32) ids[i] = key_id(W[b + i]);
                __syncwarp();
                // every row's lines are first requested into L2, a lane per row
                for (int r = lane; r < nb; r += 32) {
                    const uint8_t* rp = reinterpret_cast<const uint8_t*>(ix.vec32 + uint64_t(ids[r]) * ix.row_chunks32);
                    for (uint32_t o = 0; o < ix.row_chunks32 * 16; o += 128) prefetch_l2(rp + o);
                }
                dist32_rows(
                    ix, qs, [&](int r) { return ids[r]; }, 0, 4, nb, [&](int r, float v) { dst[r] = v; }, lane);
                __syncwarp();
                for (int i = lane; i < nb; i += 32) W[b + i] = mkkey(dst[i], ids[i]);
                __syncwarp();
            }
            for (int i = size + lane; i < a.efcap; i += 32) W[i] = ~0ull;
            __syncwarp();
#if HNSW_SORT_CHECK
            // keys are distinct (distinct ids): W needs no sort when every
            // adjacent pair is still in order
            bool unsorted = false;
            for (int i = lane; i + 1 < size; i += 32) unsorted |= W[i] > W[i + 1];
            if (__any_sync(kFull, unsorted))
#endif
                warp_sort(W, a.efcap, lane);
        }
        const int kq = a.q_kef ? int(__ldg(a.q_kef + qi) & 0xffffu) : a.k;
        const uint64_t obase = a.q_kef ? __ldg(a.q_out + qi) : uint64_t(qi) * uint64_t(a.k);
        for (int i = lane; i < kq; i += 32) {
            uint32_t oid = kNone;
            float od = __int_as_float(0x7f800000);
            if (i < size) {
                const uint64_t kk = W[i];
                oid = key_id(kk);
                od = key_dist(kk);
            }
            a.out_ids[obase + i] = oid;
            a.out_dists[obase + i] = od;
        }
        if (CHECK && bad) flags |= 4u;
        if (STOP && a.tr_count && lane == 0) a.tr_count[qi] = int(min(*n_checks, uint32_t(a.tr_max)));
        if (a.stats && lane == 0) {
            hnsw_query_stats s;
            s.n_eval = n_eval;
            s.n_exp0 = n_exp0;
            s.n_stepU = n_stepU;
            s.flags = flags;
            a.stats[qi] = s;
        }
        __syncwarp();
    }
}

}  // namespace hnswgb
