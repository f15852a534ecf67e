// fnv.cu -- the blob format's checksum (64-bit FNV-1a) on the GPU.
//
// FNV-1a is a chain over the bytes, h = (h ^ b) * p mod 2^64: one byte after
// another on the host, 0.9 ns each.  It comes apart into pieces because
//  * the low byte of h follows a chain of its own: l = ((l ^ b) * p) mod 256;
//  * h ^ b = h + ((l ^ b) - l), so with the low bytes known the chain is
//    affine: over m bytes h becomes p^m h + B, with B a function of the bytes
//    and of the low byte before them.
// Three kernels per chunk of the input:
//  fnv_maps    a warp per piece (8 KB) runs the low-byte chain from every
//              start value: 128 of them, four in a lane's two registers (16
//              bits each); start values 128 apart stay 128 apart, as the top
//              bit of l reaches no lower one.  It writes the low byte after
//              every 256 bytes, by start value.
//  fnv_starts  one block follows these maps from piece to piece.
//  fnv_pieces  a warp per piece, a lane per 256 bytes, whose low byte is now
//              known: its B, the warp's B, and the piece's share of the result.
// What bounds it: the copy of the bytes to the GPU; fnv_maps issues about 5
// instructions per byte and warp.  Measured: a 13 MB graph read, extended by
// 1,000 elements and written again, which takes two checksums: 23 ms less than
// with the host's chain (56.1 and 32.9 when it came in); a 10 MB upload 2.8 ms.
#include <cuda_runtime.h>

#include "common.hpp"
#include "index.cuh"

namespace hnswgb {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint64_t kPrime = 0x100000001b3ull;
constexpr int kSub = 256;                 // bytes of a lane
constexpr int kPiece = 32 * kSub;         // bytes of a warp
constexpr int kChunkPieces = 2048;        // 16 MB of input
constexpr int kMaps = 32 * 128;           // bytes of a piece's maps, 128 for every kSub of it
constexpr int kBatch = 256;               // pieces whose maps fnv_starts holds at a time
constexpr int kWarps = 4;

constexpr uint64_t power(uint64_t base, uint64_t n) {
    uint64_t r = 1;
    for (; n; n >>= 1, base *= base)
        if (n & 1) r *= base;
    return r;
}
constexpr uint64_t kPowSub = power(kPrime, kSub), kPowPiece = power(kPrime, kPiece);

__device__ uint64_t power_of(uint64_t base, uint32_t n) {
    uint64_t r = 1;
    for (; n; n >>= 1, base *= base)
        if (n & 1u) r *= base;
    return r;
}

struct FnvState {
    uint64_t h;    // the checksum so far
    uint32_t low;  // its low byte
};

// byte `from` of w into the low byte of both 16-bit halves
__device__ __forceinline__ uint32_t both(uint32_t w, int from) { return __byte_perm(w, 0u, 0x4040u | (from * 0x0101u)); }

// the low byte that start value l of a map (128 entries: byte 4 i + j belongs to
// value 32 j + i) leads to
__device__ __forceinline__ uint32_t follow(const uint8_t* map, uint32_t l) {
    return uint32_t(map[4 * (l & 31u) + (l >> 5 & 3u)]) ^ (l & 128u);
}

__global__ void __launch_bounds__(kWarps * 32) fnv_maps(const uint4* __restrict__ data, uint32_t pieces,
                                                        uint32_t* __restrict__ maps) {
    const int lane = threadIdx.x & 31;
    const uint32_t piece = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (piece >= pieces) return;
    const uint4* in = data + uint64_t(piece) * (kPiece / 16);
    uint32_t* out = maps + uint64_t(piece) * (kMaps / 4);
    uint32_t a = uint32_t(lane) | uint32_t(lane + 32) << 16, b = uint32_t(lane + 64) | uint32_t(lane + 96) << 16;
    uint4 next = __ldg(in);
    for (int sub = 0; sub < 32; ++sub) {
        for (int i = 0; i < kSub / 16; ++i) {
            const uint4 v = next;
            const int at = sub * (kSub / 16) + i + 1;
            next = __ldg(in + min(at, kPiece / 16 - 1));
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t x = both(w[k], j);
                    a = ((a ^ x) & 0x00ff00ffu) * uint32_t(kPrime & 0xffu);  // below 2^16 in each half
                    b = ((b ^ x) & 0x00ff00ffu) * uint32_t(kPrime & 0xffu);
                }
        }
        out[sub * 32 + lane] = __byte_perm(a, b, 0x6420);  // the low byte of each half
    }
}

// Low byte at the start of every piece; the state's h moves past the chunk
// but for the pieces' B, which fnv_pieces adds.
__global__ void __launch_bounds__(kBatch) fnv_starts(const uint32_t* __restrict__ maps, uint32_t pieces,
                                                     uint8_t* __restrict__ starts, FnvState* __restrict__ st) {
    __shared__ uint32_t m[kBatch][32];
    uint32_t low = st->low;
    for (uint32_t base = 0; base < pieces; base += kBatch) {
        const int n = int(min(uint32_t(kBatch), pieces - base));
        __syncthreads();
        for (int i = threadIdx.x; i < n * 32; i += kBatch)
            m[i >> 5][i & 31] = maps[(uint64_t(base) + (i >> 5)) * (kMaps / 4) + 31 * 32 + (i & 31)];
        __syncthreads();
        if (threadIdx.x == 0)
            for (int i = 0; i < n; ++i) {
                starts[base + i] = uint8_t(low);
                low = follow(reinterpret_cast<const uint8_t*>(m[i]), low);
            }
    }
    if (threadIdx.x == 0) {
        st->low = low;
        st->h *= power_of(kPowPiece, pieces);
    }
}

__global__ void __launch_bounds__(kWarps * 32) fnv_pieces(const uint4* __restrict__ data, uint32_t pieces,
                                                          const uint8_t* __restrict__ maps,
                                                          const uint8_t* __restrict__ starts,
                                                          FnvState* __restrict__ st) {
    const int lane = threadIdx.x & 31;
    const uint32_t piece = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (piece >= pieces) return;
    uint32_t l = starts[piece];
    if (lane > 0) l = follow(maps + uint64_t(piece) * kMaps + uint32_t(lane - 1) * 128, l);
    const uint4* in = data + uint64_t(piece) * (kPiece / 16) + lane * (kSub / 16);
    uint64_t h = l;
    for (int i = 0; i < kSub / 16; ++i) {
        const uint4 v = __ldg(in + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < 4; ++j) h = (h ^ (w[k] >> (8 * j) & 0xffu)) * kPrime;
    }
    uint64_t B = (h - kPowSub * l) * power_of(kPowSub, uint32_t(31 - lane));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) B += __shfl_xor_sync(kFull, B, o);
    if (lane == 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(&st->h), B * power_of(kPowPiece, pieces - 1 - piece));
}

// Below this the launches and the copy cost as much as the host's chain
// (256 KB: 0.24 ms on the host).
constexpr uint64_t kMinBytes = 256 << 10;

bool on_gpu(const uint8_t* p, uint64_t n, cudaStream_t s, uint64_t& out) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return false;
    const uint64_t pieces = n / kPiece;
    const uint64_t most = pieces < uint64_t(kChunkPieces) ? pieces : uint64_t(kChunkPieces);
    // from the pool as the process has set it up: by default the memory goes
    // back at the synchronisation below
    void* scr = nullptr;
    if (cudaMallocAsync(&scr, most * (kPiece + kMaps) + 256 + most, s) != cudaSuccess) return false;
    uint8_t* data = static_cast<uint8_t*>(scr);
    uint8_t* maps = data + most * kPiece;
    FnvState* st = reinterpret_cast<FnvState*>(maps + most * kMaps);
    uint8_t* starts = maps + most * kMaps + 256;
    FnvState host{kFnvBasis, uint32_t(kFnvBasis & 0xffu)};
    cudaError_t e = cudaMemcpyAsync(st, &host, sizeof(host), cudaMemcpyHostToDevice, s);
    for (uint64_t at = 0; at < pieces && e == cudaSuccess; at += most) {
        const uint32_t m = uint32_t(pieces - at < most ? pieces - at : most);
        e = cudaMemcpyAsync(data, p + at * kPiece, uint64_t(m) * kPiece, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) break;
        const unsigned blocks = (m + kWarps - 1) / kWarps;
        fnv_maps<<<blocks, kWarps * 32, 0, s>>>(reinterpret_cast<const uint4*>(data), m,
                                                reinterpret_cast<uint32_t*>(maps));
        fnv_starts<<<1, kBatch, 0, s>>>(reinterpret_cast<const uint32_t*>(maps), m, starts, st);
        fnv_pieces<<<blocks, kWarps * 32, 0, s>>>(reinterpret_cast<const uint4*>(data), m, maps, starts, st);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&host, st, sizeof(host), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(scr, s);
    const cudaError_t done = cudaStreamSynchronize(s);  // also after a failure: p may still be read
    if (e != cudaSuccess || done != cudaSuccess) return false;
    out = fnv1a64(p + pieces * kPiece, n - pieces * kPiece, host.h);
    return true;
}

}  // namespace

uint64_t checksum64(const uint8_t* p, uint64_t n, cudaStream_t s) {
    if (n >= kMinBytes) {
        uint64_t h = 0;
        if (on_gpu(p, n, s, h)) return h;
        cudaGetLastError();  // no device, or no memory on it: the host's chain
    }
    return fnv1a64(p, n);
}

}  // namespace hnswgb
