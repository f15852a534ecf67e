// search_dev.cuh -- device code shared by the search kernels (search.cu: one
// warp per query; search_team.cuh: a block per query): launch arguments, keys,
// row decoding and distances, the visited set, the merges into W, rerank.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>
#include <cstring>

#include "index.cuh"
#include "stopnet.cuh"

namespace hnswgb {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxNbr = 64;  // neighbour slots of an element on a layer (Mmax0 and Mmax <= 64)

// Tuning switches (compile time).  HNSW_PREFETCH_ROWS: after the visited
// check, every lane owning a new neighbour prefetches its whole row into L2,
// so the later gather rounds of the batch hit L2 instead of waiting on DRAM
// one after another.  HNSW_PREFETCH_NEXT: while an element is expanded, the
// neighbour row of the next unexpanded entry of W is loaded speculatively;
// it is the next element to expand unless the current batch inserts a better
// one.
#ifndef HNSW_PREFETCH_ROWS
#define HNSW_PREFETCH_ROWS 0
#endif
#ifndef HNSW_PREFETCH_NEXT
#define HNSW_PREFETCH_NEXT 1
#endif
// HNSW_STOP_SKIP_IMPROVING: outside trace recording, a due check is put off
// while the expansion just done changed the K nearest of W (the search is
// still improving its answer), to the first later expansion that does not
#ifndef HNSW_STOP_SKIP_IMPROVING
#define HNSW_STOP_SKIP_IMPROVING 1
#endif
// HNSW_STOP_NOINLINE: the stop check (features + network) as a called
// function instead of inline code in the layer-0 loop
#ifndef HNSW_STOP_NOINLINE
#define HNSW_STOP_NOINLINE 0
#endif
#if HNSW_STOP_NOINLINE
#define HNSW_STOP_FN __device__ __noinline__
#else
#define HNSW_STOP_FN __device__ __forceinline__
#endif
// rows gathered per team and round for fp32 rows of 128 coordinates and for
// bf16/f16 rows of up to 128 coordinates
#ifndef HNSW_F32_U
#define HNSW_F32_U 2
#endif
#ifndef HNSW_B16_U
#define HNSW_B16_U 2
#endif
// HNSW_FP8_U: rows a team of fp8 rows keeps in flight (2: 64 registers,
// 32 warps per SM; 8 took 96 registers, 20 warps, and ran 1.7x slower)
#ifndef HNSW_FP8_U
#define HNSW_FP8_U 2
#endif
// HNSW_F16_U: the same for f16 rows (2: 64 registers; 4 took 80 registers
// and ran 1.2x slower)
#ifndef HNSW_F16_U
#define HNSW_F16_U 2
#endif
// HNSW_MERGE_BALLOT: a merge with at most HNSW_MERGE_BALLOT_MAX candidates
// finds their places in W by ballots over the entries held in registers
// instead of a binary search
#ifndef HNSW_MERGE_BALLOT
#define HNSW_MERGE_BALLOT 1
#endif
#ifndef HNSW_MERGE_BALLOT_MAX
#define HNSW_MERGE_BALLOT_MAX 3
#endif
// HNSW_SORT_CHECK: after the rerank, W is sorted only when some adjacent
// pair is out of order
#ifndef HNSW_SORT_CHECK
#define HNSW_SORT_CHECK 1
#endif
// HNSW_MIXED_SUB: for bf16 / f16 rows and squared L2, x - q in one
// mixed-precision subtraction per coordinate (the 16-bit x taken as it is
// stored, q in fp32, the difference rounded once to fp32: the same value as
// decoding x to fp32 and subtracting)
#ifndef HNSW_MIXED_SUB
#define HNSW_MIXED_SUB 1
#endif

// x - q for the two 16-bit values of w (low half first), rounded once to fp32
template <int ST>
__device__ __forceinline__ void sub_halves(uint32_t w, float q0, float q1, float& t0, float& t1) {
    if (ST == HNSW_BF16)
        asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n sub.rn.f32.bf16 %0, l, %3;\n sub.rn.f32.bf16 %1, h, %4;\n}"
            : "=f"(t0), "=f"(t1) : "r"(w), "f"(q0), "f"(q1));
    else
        asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n sub.rn.f32.f16 %0, l, %3;\n sub.rn.f32.f16 %1, h, %4;\n}"
            : "=f"(t0), "=f"(t1) : "r"(w), "f"(q0), "f"(q1));
}

struct SearchArgs {
    DevIndex ix;
    const float* q;
    uint32_t n;
    int k;
    int efp;
    int efcap;      // power of two >= efp
    int hlog;       // log2 visited slots
    int warp_smem;  // bytes of shared memory per warp
    // per-warp layout: W, the visited set, ids, dst, nbuf (kMaxNbr entries
    // each) and aux (64 bytes) at fixed places, then at these byte offsets
    // from the warp's region: hs (the stop check's scratch, learned-stop
    // launches only) and qs (the rerank's copy of q, in the visited set's
    // bytes when they suffice: it is filled after the search)
    int off_hs, off_qs;
    int rerank;
    uint32_t* out_ids;
    float* out_dists;
    hnsw_query_stats* stats;
    uint32_t* work;
    // learned stop: model (null: none), decision threshold on the logit,
    // check period in layer-0 expansions (0: no checks)
    const StopDev* stop;
    float stop_logit;
    int stop_period;
    // trace mode (tr_count != null): record every check, never stop early
    float* tr_feat;      // [n][tr_max][6]
    uint32_t* tr_topk;   // [n][tr_max][k]
    float* tr_logit;     // [n][tr_max] (only with a model)
    int32_t* tr_count;   // [n] checks recorded
    int tr_max;
    // grouped launch (several requests in one launch): per-query k (low 16
    // bits) and ef (high 16 bits), and the first output slot of each query;
    // null: k, efp and qi * k for every query
    const uint32_t* q_kef;
    const uint64_t* q_out;
    // two-pass scheduling: mode 0 = descent and beam per query in input order;
    // mode 1 = descent only, writing the layer-0 enter key and the upper-layer
    // counters of every query; mode 2 = beam only, queries taken in `order`
    int mode;
    uint64_t* ep_keys;   // [n]
    uint32_t* up_cnt;    // [n][2]: distance evaluations, rows read on layers >= 1
    const uint32_t* order;
    // deferral (mode 0, null: off): a query whose descent ends nearer than
    // the mean descent distance of the queries before it is pushed, with its
    // layer-0 enter key and upper-layer counters, and its beam runs once the
    // input queue is drained, so that the far (long) searches start first.
    // dfr_ctl: [0] records pushed, [1] claim tickets taken, [2] error (a
    // record that never appeared), [3] descents seen, [4] their distance sum
    // (fp32), [5] input-queue queries past their decision.
    // dfr_rec[i]: enter key low / high word, counters (rows read on layers
    // >= 1 << 20 | distance evaluations), query index -- written last, all
    // ones until then.
    uint32_t* dfr_ctl;
    uint4* dfr_rec;  // [n]
    int dfr_hold;    // test hook: query 0's decision is never counted
    // block-per-query kernel (search_team.cuh): byte offsets of its pieces in
    // the block's shared memory
    int off_vis, off_slot, off_merge, off_ctl;
    uint32_t* err;   // the index's error word (host memory mapped on the device)
};

// What a launch asks of the instantiations of its storage type.
struct KernelAsk {
    uint32_t chunks;  // 16-byte chunks per stored row
    bool stop;        // learned-stop checks or trace recording
    bool wide;        // W of more than 64 entries, or layer-0 lists of more than 32
    bool check;       // the bounds-checked build
    int team_r;       // a block per query with W in 2, 8 or 16 registers per lane (0: a warp per query)
};
using KernelFn = void (*)(const SearchArgs);
// the instantiation, or null when the format has none (search_f32.cu, ...)
KernelFn search_kernel_f32(const KernelAsk& k);
KernelFn search_kernel_bf16(const KernelAsk& k);
KernelFn search_kernel_f16(const KernelAsk& k);
KernelFn search_kernel_fp8(const KernelAsk& k);

// ---- keys -----------------------------------------------------------------
// key = ord(dist) << 32 | id << 1 | expanded.  key >> 1 orders (dist, id).
// The bits are taken by an instruction of its own: where the compiler sees that
// f is a sum of squares it takes the sign bit for clear and makes the flip a
// float negation, which gives a NaN back without its sign -- a key below all
// others instead of above them, and a distance of -0.
__device__ __forceinline__ uint32_t f2ord(float f) {
    uint32_t b;
    asm("mov.b32 %0, %1;" : "=r"(b) : "f"(f));
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t o) {
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}
__device__ __forceinline__ uint64_t mkkey(float d, uint32_t id) {
    return (uint64_t(f2ord(d)) << 32) | (uint64_t(id) << 1);
}
__device__ __forceinline__ uint32_t key_id(uint64_t k) { return uint32_t(k >> 1) & 0x7fffffffu; }
__device__ __forceinline__ float key_dist(uint64_t k) { return ord2f(uint32_t(k >> 32)); }

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) {
    const uint32_t hi = uint32_t(v >> 32), lo = uint32_t(v);
    const uint32_t mh = __reduce_min_sync(kFull, hi);
    const uint32_t ml = __reduce_min_sync(kFull, hi == mh ? lo : 0xffffffffu);
    return (uint64_t(mh) << 32) | ml;
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// 16-byte asynchronous global -> shared copy (no registers held while in flight)
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Row gathers are random and not reused by this SM: keep them out of L1 so
// that L1 holds what is reused (the stop network's weights).
#ifndef HNSW_ROW_NO_L1
#define HNSW_ROW_NO_L1 0
#endif
__device__ __forceinline__ uint4 ld_row_chunk(const uint4* p) {
    uint4 v;
#if HNSW_ROW_NO_L1
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
#else
    asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
#endif
    return v;
}

// ---- storage decoding -----------------------------------------------------
template <int ST>
struct Store;
template <>
struct Store<HNSW_F32> {
    static constexpr int CPC = 4;
    __device__ static void decode(const uint4& v, float* x) {
        x[0] = __uint_as_float(v.x); x[1] = __uint_as_float(v.y);
        x[2] = __uint_as_float(v.z); x[3] = __uint_as_float(v.w);
    }
};
template <>
struct Store<HNSW_BF16> {
    static constexpr int CPC = 8;
    __device__ static void decode(const uint4& v, float* x) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
};
template <>
struct Store<HNSW_F16> {
    static constexpr int CPC = 8;
    __device__ static void decode(const uint4& v, float* x) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __half2 h;
            memcpy(&h, &w[i], 4);
            const float2 f = __half22float2(h);
            x[2 * i] = f.x;
            x[2 * i + 1] = f.y;
        }
    }
};
template <>
struct Store<HNSW_FP8E4M3> {
    static constexpr int CPC = 16;
    __device__ static void decode(const uint4& v, float* x) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const __nv_fp8x2_storage_t pr = __nv_fp8x2_storage_t((w[i] >> (16 * j)) & 0xffffu);
                const __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2(pr, __NV_E4M3);
                __half2 h;
                memcpy(&h, &hr, 4);
                const float2 f = __half22float2(h);
                x[4 * i + 2 * j] = f.x;
                x[4 * i + 2 * j + 1] = f.y;
            }
        }
    }
};

// ---- batched distance of n rows -------------------------------------------
// FULL: every row has exactly TEAM * CPL chunks (no per-chunk bounds test)
template <int ST, int TEAM, int CPL, int U, bool FULL>
struct Dist {
    static constexpr int CPC = Store<ST>::CPC;
    static constexpr int QF = CPL * CPC;  // query coordinates held per lane
    static constexpr int TEAMS = 32 / TEAM;
    static constexpr int RPR = TEAMS * U;  // rows per round
    static_assert(U <= TEAM, "the joint reduction halves a team per halving of its rows");
    static constexpr bool MIXED = HNSW_MIXED_SUB && (ST == HNSW_BF16 || ST == HNSW_F16);

    __device__ static void load_q(const float* qp, uint32_t d, float (&qr)[QF], int lane) {
        const int tl = lane % TEAM;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int ch = tl + c * TEAM;
#pragma unroll
            for (int j = 0; j < CPC; ++j) {
                const uint32_t co = uint32_t(ch * CPC + j);
                qr[c * CPC + j] = co < d ? qp[co] : 0.0f;
            }
        }
    }

    // A lane's share of one row's sum: the chunks v it read of the row.
    __device__ static float share(const float (&qr)[QF], const uint4 (&v)[CPL], float sc, bool l2) {
        float acc = 0.0f;
        if (MIXED && l2) {
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const uint32_t w[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float t0, t1;
                    sub_halves<ST>(w[i], qr[c * CPC + 2 * i], qr[c * CPC + 2 * i + 1], t0, t1);
                    acc = fmaf(t0, t0, acc);
                    acc = fmaf(t1, t1, acc);
                }
            }
            return acc;
        }
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            float x[CPC];
            Store<ST>::decode(v[c], x);
#pragma unroll
            for (int j = 0; j < CPC; ++j) {
                const float xv = ST == HNSW_FP8E4M3 ? x[j] * sc : x[j];
                if (l2) {
                    const float t = qr[c * CPC + j] - xv;
                    acc = fmaf(t, t, acc);
                } else {
                    acc = fmaf(qr[c * CPC + j], xv, acc);
                }
            }
        }
        return acc;
    }

    // run() where the warp takes one row at a time (rows above 128 coordinates):
    // written out so that the reads of two rows overlap (10,000 queries at ef
    // 50, a row after another / so: 200 fp32 coordinates 854 / 810 us, 256 bf16
    // 687 / 649, 256 fp8 735 / 722; the fp8 instances with the stop then spill 8
    // to 40 bytes and are as quick or quicker all the same)
    __device__ static void run_row_pairs(const DevIndex& ix, const float (&qr)[QF], const uint32_t* ids, int n,
                                         float* out, int lane) {
        const uint32_t C = ix.row_chunks;
        const bool l2 = ix.metric == HNSW_L2SQ;
#pragma unroll 2
        for (int r = 0; r < n; ++r) {
            const uint4* rowp = ix.vec + uint64_t(ids[r]) * C;
            uint4 v[CPL];
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const uint32_t ch = uint32_t(lane + c * 32);
                v[c] = FULL || ch < C ? ld_row_chunk(rowp + ch) : make_uint4(0u, 0u, 0u, 0u);
            }
            float sc = 0.0f;
            if (ST == HNSW_FP8E4M3) sc = __ldg(ix.scale + ids[r]);
            float acc = share(qr, v, sc, l2);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
            if (lane == 0) out[r] = l2 ? acc : 1.0f - acc;
        }
    }

    // out[r] = distance(q, row ids[r]) for r < n.  The search is bound by
    // instruction issue as much as by the gathers, so a row costs as few
    // instructions as it can: a team past the end reads the last row again
    // instead of clearing its registers, a turn in which no team has a row is
    // skipped, and the U sums of a team are reduced together -- at each step
    // of the butterfly half of the lanes go on with half of the rows, which
    // halves the shuffles; every sum adds the same pairs in the same order as
    // a butterfly of its own.  Measured per 10,000 queries on SIFT-shaped 1M
    // at ef 50 (bf16 + rerank / fp32): 600 / 628 us before, 550 / 587 with
    // plain reductions, 520 / 575 us with joint ones.
    __device__ static void run(const DevIndex& ix, const float (&qr)[QF], const uint32_t* ids, int n,
                               float* out, int lane) {
        if constexpr (TEAM == 32 && U == 1) {
            run_row_pairs(ix, qr, ids, n, out, lane);
            return;
        }
        const int team = lane / TEAM, tl = lane % TEAM;
        const uint32_t C = ix.row_chunks;
        for (int base = 0; base < n; base += RPR) {
            uint4 v[U][CPL];
            float sc[U] = {}, acc[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                // a team past the end reads the last row once more
                const uint32_t id = ids[min(base + u * TEAMS + team, n - 1)];
                const uint4* rowp = ix.vec + uint64_t(id) * C;
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    const uint32_t ch = uint32_t(tl + c * TEAM);
                    if (FULL || ch < C)
                        v[u][c] = ld_row_chunk(rowp + ch);
                    else
                        v[u][c] = make_uint4(0u, 0u, 0u, 0u);
                }
                if (ST == HNSW_FP8E4M3) sc[u] = __ldg(ix.scale + id);
            }
            const bool l2 = ix.metric == HNSW_L2SQ;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                acc[u] = 0.0f;
                if (u == 0 || base + u * TEAMS < n) acc[u] = share(qr, v[u], sc[u], l2);
            }
            int u = 0, cnt = U, lvl = 0;  // u: the row whose sum this lane ends with
#pragma unroll
            for (int o = TEAM / 2; o > 0; o >>= 1) {
                if (cnt > 1) {
                    cnt >>= 1;
                    const bool up = (tl & o) != 0;
                    u += int(up) << lvl++;
#pragma unroll
                    for (int i = 0; i < cnt; ++i) {
                        const float other = up ? acc[2 * i] : acc[2 * i + 1];
                        acc[i] = (up ? acc[2 * i + 1] : acc[2 * i]) + __shfl_xor_sync(kFull, other, o);
                    }
                } else {
                    acc[0] += __shfl_xor_sync(kFull, acc[0], o);
                }
            }
            const int r = base + u * TEAMS + team;
            if (tl % (TEAM / U) == 0 && r < n) out[r] = l2 ? acc[0] : 1.0f - acc[0];
        }
    }
};

// exact fp32 distances from the fp32 copy (rerank) of rows first, first + 1,
// ..., then step further, up to n (row r is element id(r); out(r, distance)
// is called on one lane): teams of 8 lanes take a row each, 4 rows per warp
// round, every chunk a lane reads of its row (up to 32 chunks per pass)
// loaded before any is used; q in shared memory
template <class Id, class Out>
__device__ __forceinline__ void dist32_rows(const DevIndex& ix, const float* qs, Id id, int first, int step, int n,
                                            Out out, int lane) {
    const int team = lane >> 3, tl = lane & 7;
    const uint32_t C = ix.row_chunks32;
    const float4* q4 = reinterpret_cast<const float4*>(qs);
    for (int base = first; base < n; base += step) {
        const int r = base + team;
        const bool live = r < n;
        const uint4* rowp = ix.vec32 + uint64_t(live ? id(r) : 0u) * C;
        float acc = 0.0f;
        for (uint32_t cb = 0; cb < C; cb += 32) {
            uint4 v[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t ch = cb + uint32_t(tl + 8 * c);
                v[c] = (live && ch < C) ? ld_row_chunk(rowp + ch) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t ch = cb + uint32_t(tl + 8 * c);
                if (ch >= C) break;
                const float4 qq = q4[ch];
                const float qv[4] = {qq.x, qq.y, qq.z, qq.w};
                const float x[4] = {__uint_as_float(v[c].x), __uint_as_float(v[c].y), __uint_as_float(v[c].z),
                                    __uint_as_float(v[c].w)};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (ix.metric == HNSW_L2SQ) {
                        const float t = qv[j] - x[j];
                        acc = fmaf(t, t, acc);
                    } else {
                        acc = fmaf(qv[j], x[j], acc);
                    }
                }
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
        if (tl == 0 && live) out(r, ix.metric == HNSW_L2SQ ? acc : 1.0f - acc);
    }
}

// ---- visited set ------------------------------------------------------------
// 4-way bucketed hash of element ids: one 16-byte shared load reads a whole
// bucket; a miss stores the id into the bucket's first empty slot, or, when
// the bucket is full, over slot (id & 3) -- the set then forgets that slot's
// element (harmless, see the file header).  Two lanes of a warp inserting
// into the same slot at once lose one of the ids the same way.
// Returns true when `id` was not in the set (and records it).
__device__ __forceinline__ bool visit_new(uint32_t* H, int hlog, uint32_t id, uint32_t& flags) {
    const uint32_t b = (id * 2654435761u) >> (34 - hlog);  // bucket index, 2^(hlog-2) buckets
    uint4* bp = reinterpret_cast<uint4*>(H) + b;
    const uint4 v = *bp;
    if (v.x == id || v.y == id || v.z == id || v.w == id) return false;
    uint32_t* sl = reinterpret_cast<uint32_t*>(bp);
    int slot = v.x == kNone ? 0 : (v.y == kNone ? 1 : (v.z == kNone ? 2 : (v.w == kNone ? 3 : -1)));
    if (slot < 0) {
        slot = int(id & 3u);
        flags |= 1u;
    }
    sl[slot] = id;
    return true;
}

// Both merges take a new key per lane (ok: this lane has one; keys of elements
// not in W yet, or repeated ones, which are dropped) and leave in W the efp
// smallest keys of W and the new ones, in order -- the result of Alg. 2's
// admissions and evictions one at a time.  They return the smallest index
// that received a new key (INT_MAX: none did); ok stays set in the lanes whose
// key is now in W.

// W of at most 64 entries, or up to kNarrow ones of a longer beam's W (whose
// lower bounds reach 63).  Every surviving key finds its lower bound in W by
// ballots (few candidates) or a binary search of its own; one pass over the
// survivors then gives each its rank among them (its final position is lower
// bound + rank) and each W entry the number of survivors placed before it; W
// is read into registers (entries lane and lane + 32) before any write, and
// every entry is written once.
constexpr int kNarrow = 63;
__device__ __forceinline__ int merge_small(uint64_t* W, int& size, int efp, uint64_t k, bool& ok, int lane) {
    // W's entries lane and lane + 32 (beyond size: all ones, above every key)
    const uint64_t w0 = lane < size ? W[lane] : ~0ull;
    const uint64_t w1 = lane + 32 < size ? W[lane + 32] : ~0ull;
    const bool full = size >= efp;
    const uint64_t wlast = size > 0 ? (W[size - 1] >> 1) : 0ull;
    const uint64_t k1 = k >> 1;
    ok = ok && !(full && k1 > wlast);
    int lb = 0;
    const uint32_t cand = __ballot_sync(kFull, ok);
    if (cand == 0) return INT_MAX;
    int rank = 0, c0 = 0, c1 = 0;  // survivors below my key; placed before my W entries
    uint32_t surv = 0;
#if HNSW_MERGE_BALLOT
    if (__popc(cand) <= HNSW_MERGE_BALLOT_MAX) {
        // few candidates: each one's lower bound and duplicate test by
        // ballots over the entries held in registers (a new key has the
        // expanded bit clear: an entry is below it, bit or no bit, when its
        // whole word is; the same element is the same low word but for that
        // bit), and its effect on the ranks and the entries' moves in the
        // same turn
        for (uint32_t bits = cand; bits; bits &= bits - 1) {
            const int sl = __ffs(bits) - 1;
            const uint64_t ks = __shfl_sync(kFull, k, sl);
            const uint32_t id1 = uint32_t(ks) | 1u;
            if (__any_sync(kFull, (uint32_t(w0) | 1u) == id1 || (uint32_t(w1) | 1u) == id1)) continue;  // already in W
            surv |= 1u << sl;
            const bool b0 = w0 < ks, b1 = w1 < ks;
            const int l = __popc(__ballot_sync(kFull, b0)) + __popc(__ballot_sync(kFull, b1));
            if (lane == sl) lb = l;
            c0 += !b0;
            c1 += !b1;
            rank += ks < k;
        }
        if (surv == 0) return INT_MAX;
        ok = (surv >> lane) & 1u;
    } else
#endif
    {
        if (ok) {
#pragma unroll
            for (int step = 32; step > 0; step >>= 1)  // entries of W below k1
                if (lb + step <= size && (W[lb + step - 1] >> 1) < k1) lb += step;
            if (lb < size && (W[lb] >> 1) == k1) ok = false;  // already in W
        }
        surv = __ballot_sync(kFull, ok);
        if (surv == 0) return INT_MAX;
        for (uint32_t bits = surv; bits; bits &= bits - 1) {
            const int sl = __ffs(bits) - 1;
            const uint64_t ks = __shfl_sync(kFull, k1, sl);
            const int ls = __shfl_sync(kFull, lb, sl);
            rank += ks < k1;
            c0 += ls <= lane;
            c1 += ls <= lane + 32;
        }
    }
    __syncwarp();
    if (lane < size && lane + c0 < efp) W[lane + c0] = w0;
    if (lane + 32 < size && lane + 32 + c1 < efp) W[lane + 32 + c1] = w1;
    int pos = INT_MAX;
    if (ok) {
        pos = lb + rank;
        ok = pos < efp;
        if (ok)
            W[pos] = k;
        else
            pos = INT_MAX;
    }
    size = min(efp, size + __popc(surv));
    __syncwarp();
    return int(__reduce_min_sync(kFull, uint32_t(pos)));
}

// W of up to 1,024 entries.  Lower bounds by ballots (BALLOT: where registers
// are left for them) or binary search, ranks among the survivors as above; the
// final positions of the new keys are then a bitmap (one 32-bit word per lane:
// 1,024 positions); the count of its bits below a position says where that
// position's entry comes from, so that W moves up in one pass over its 32-entry
// chunks, top chunk first, with a few instructions per chunk whatever the number
// of new keys.  The form that counted, for every entry, the new keys placed
// before it took a pass over the new keys per chunk: GloVe-shaped 400k, 10,000
// queries at ef 498: 7.19 ms, 5.85 ms with this merge and the shorter row
// distances.  A single new key needs no bitmap.  That, and merge_small while W
// is short, is for beams just above 64 entries, where most of a search is W's
// growth and single keys: SIFT-shaped 1M, 1,200 queries at ef 66, us with the
// counting form / without these two / with them: f16 529 / 542 / 532, fp32 535 /
// 550 / 536.
template <bool BALLOT>
__device__ __forceinline__ int merge_wide(uint64_t* W, int& size, int efp, uint64_t k, bool& ok, int lane) {
    const uint64_t wlast = size > 0 ? (W[size - 1] >> 1) : 0ull;
    const uint64_t k1 = k >> 1;
    ok = ok && !(size >= efp && k1 > wlast);
    const uint32_t cand = __ballot_sync(kFull, ok);
    if (cand == 0) return INT_MAX;
    int lb = 0;
    if (BALLOT && __popc(cand) <= HNSW_MERGE_BALLOT_MAX) {
        // few candidates: the 32 entries that hold the place by a ballot over
        // the last entries of all 32s, the place by one over these (two reads
        // of shared memory in a row instead of up to ten)
        const uint64_t top = 32 * lane < size ? W[min(32 * lane + 31, size - 1)] : ~0ull;
        for (uint32_t bits = cand; bits; bits &= bits - 1) {
            const int sl = __ffs(bits) - 1;
            const uint64_t ks = __shfl_sync(kFull, k, sl);  // expanded bit clear
            const int base = 32 * __popc(__ballot_sync(kFull, top < ks));
            const uint64_t v = base + lane < size ? W[base + lane] : ~0ull;
            const int l = min(base + __popc(__ballot_sync(kFull, v < ks)), size);
            const bool dup = __any_sync(kFull, (v | 1ull) == (ks | 1ull));  // already in W
            if (lane == sl) {
                lb = l;
                ok = !dup;
            }
        }
    } else if (ok) {
        for (int step = 1 << (31 - __clz(size | 1)); step > 0; step >>= 1)  // entries of W below k1
            if (lb + step <= size && (W[lb + step - 1] >> 1) < k1) lb += step;
        if (lb < size && (W[lb] >> 1) == k1) ok = false;  // already in W
    }
    const uint32_t surv = __ballot_sync(kFull, ok);
    if (surv == 0) return INT_MAX;
    if (!(surv & (surv - 1))) {  // one new key, the common case in a full W: its place is known
        const int p = __shfl_sync(kFull, lb, __ffs(surv) - 1);
        const int nsize = min(efp, size + 1);
        for (int c = (nsize - 1) >> 5; c >= p >> 5; --c) {
            const int t = c * 32 + lane;
            const bool mv = t > p && t < nsize;
            const uint64_t v = mv ? W[t - 1] : 0ull;
            __syncwarp();  // a chunk's reads precede its writes
            if (mv) W[t] = v;
        }
        if (ok) W[p] = k;
        size = nsize;
        __syncwarp();
        return p;
    }
    int pos = lb;
    for (uint32_t bits = surv; bits; bits &= bits - 1) pos += __shfl_sync(kFull, k1, __ffs(bits) - 1) < k1;
    ok = ok && pos < efp;
    const uint32_t in = __ballot_sync(kFull, ok);  // not empty: the smallest survivor is below W's last entry
    const int first = int(__reduce_min_sync(kFull, ok ? uint32_t(pos) : 0xffffffffu));
    const int nsize = min(efp, size + __popc(surv));
    uint32_t word = 0;  // new keys' positions lane * 32 .. lane * 32 + 31
    for (uint32_t bits = in; bits; bits &= bits - 1) {
        const int p = __shfl_sync(kFull, pos, __ffs(bits) - 1);
        if ((p >> 5) == lane) word |= 1u << (p & 31);
    }
    int below = __popc(in);  // new positions below the chunk
    for (int c = (nsize - 1) >> 5; c >= first >> 5; --c) {
        const uint32_t wc = __shfl_sync(kFull, word, c);
        below -= __popc(wc);
        const int t = c * 32 + lane;
        const int src = t - below - __popc(wc & lanemask_lt());
        const bool mv = !((wc >> lane) & 1u) && t > first && t < nsize;
        const uint64_t v = mv ? W[src] : 0ull;
        __syncwarp();  // a chunk's reads (at most this chunk's positions) precede its writes
        if (mv) W[t] = v;
    }
    if (ok) W[pos] = k;
    size = nsize;
    __syncwarp();
    return first;
}
// warp-wide bitonic sort of n (power of two) keys in shared memory
inline __device__ void warp_sort(uint64_t* a, int n, int lane) {
    for (int kk = 2; kk <= n; kk <<= 1)
        for (int j = kk >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < n; i += 32) {
                const int p = i ^ j;
                if (p > i) {
                    const uint64_t x = a[i], y = a[p];
                    const bool up = (i & kk) == 0;
                    if ((x > y) == up) {
                        a[i] = y;
                        a[p] = x;
                    }
                }
            }
            __syncwarp();
        }
}

}  // namespace hnswgb
