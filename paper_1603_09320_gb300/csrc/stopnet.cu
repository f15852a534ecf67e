// stopnet.cu -- training of the learned early-stop network on the GPU and
// its upload into an index (hnsw_stop_grad, hnsw_stop_train,
// hnsw_set_stop_model, hnsw_clear_stop_model).  The paper has no counterpart.
//
// Training is mini-batch gradient descent on the mean binary cross-entropy
// of sigmoid(logit) against the 0/1 labels, with Adam (fp32 master weights,
// fp16 working weights: the forward and backward passes use the fp16 values,
// as inference does).  A block runs the forward and backward pass of tiles of
// 32 samples with all activations in shared memory and writes its partial
// sum of the gradient; an optimiser kernel adds the blocks' sums in order and
// updates the weights (so a run's result is a function of its inputs alone).
// Samples are visited in a different affine order each epoch.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "common.hpp"
#include "index.cuh"
#include "stopnet.cuh"

namespace hnswgb {
namespace {

constexpr int kTB = 32;        // samples per tile
constexpr int kThreads = 256;
constexpr int kLd = kStopH + 4;  // padded row of the activation and weight tiles (16-byte aligned)
constexpr int kPartLd = (kStopParams + 1 + 31) / 32 * 32;  // a block's partial sums: gradient, loss, padding

struct TrainSmem {
    float w2[kStopH * kLd], w2t[kStopH * kLd];  // W2 by output row, and by input row
    float w1[kStopH * kStopIn], b1[kStopH], b2[kStopH], w3[kStopH];
    float h1[kTB * kLd];  // relu(a1)
    float a2[kTB * kLd];
    float d2[kTB * kLd];  // d(loss)/d(a2)
    float d1[kTB * kLd];  // d(loss)/d(a1)
    float x[kTB * kStopIn], y[kTB], dz[kTB], ls[kTB];
    float mu[kStopIn], isig[kStopIn];
    int idx[kTB];
};

__device__ __forceinline__ int sample_index(int64_t i, int64_t n, uint64_t a, uint64_t c) {
    return int((a * uint64_t(i) + c) % uint64_t(n));
}

// Consecutive kernels of a training run are launched with programmatic
// serialisation: a kernel may start while the one before it drains, and waits
// here, before it reads anything that one writes, until that one has ended
// and its writes are visible; such values are read from L2 (__ldcg): a line in
// L1 may be older than the wait.
__device__ __forceinline__ void wait_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ float ld_weight(const __half* p) {
    __half_raw r;
    r.x = __ldcg(reinterpret_cast<const unsigned short*>(p));
    return __half2float(__half(r));
}

// out[b0..b0+1][c0..c0+3] of A [kTB][64] times B [64][64] (rows kLd apart)
__device__ __forceinline__ void tile_2x4(const float* A, const float* B, int b0, int c0, float (&o)[2][4]) {
#pragma unroll 4
    for (int k = 0; k < kStopH; k += 4) {
        const float4 a0 = *reinterpret_cast<const float4*>(A + b0 * kLd + k);
        const float4 a1 = *reinterpret_cast<const float4*>(A + (b0 + 1) * kLd + k);
        const float p[4] = {a0.x, a0.y, a0.z, a0.w}, q[4] = {a1.x, a1.y, a1.z, a1.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 b = *reinterpret_cast<const float4*>(B + (k + i) * kLd + c0);
            o[0][0] = fmaf(p[i], b.x, o[0][0]);
            o[0][1] = fmaf(p[i], b.y, o[0][1]);
            o[0][2] = fmaf(p[i], b.z, o[0][2]);
            o[0][3] = fmaf(p[i], b.w, o[0][3]);
            o[1][0] = fmaf(q[i], b.x, o[1][0]);
            o[1][1] = fmaf(q[i], b.y, o[1][1]);
            o[1][2] = fmaf(q[i], b.z, o[1][2]);
            o[1][3] = fmaf(q[i], b.w, o[1][3]);
        }
    }
}

// Forward + backward of samples [base, end) of the epoch order; the block's
// sums of scale * gradient and scale * loss go to its row of part.
//
// A step of 4,096 samples is 55 MFMA: two microseconds of the chip when it is
// spread over it.  Tiles of 32 samples give such a step 128 blocks (128-sample
// tiles: 32, on 152 SMs), every 64-wide product is tiled in registers (2x4
// outputs per thread forward and through W2, 4x4 of W2's gradient, fed by
// 16-byte shared loads; scalar loads, two per multiply-add, took 80 us a step),
// the gradient stays in registers over a block's tiles, and blocks write
// partial sums instead of adding into one buffer: 4,673 atomics per block, and
// an order of addition that changed from run to run.  Measured, 200,000
// samples, 2 epochs (98 steps): 9.2 ms before, 1.7 ms now.
__global__ void __launch_bounds__(kThreads) stop_fwd_bwd(const float* __restrict__ X, const float* __restrict__ Y,
                                                         int64_t n, uint64_t pa, uint64_t pc, int64_t base, int64_t end,
                                                         const float* __restrict__ norm,
                                                         const __half* __restrict__ w, float* __restrict__ part,
                                                         float scale) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(sm_raw);
    const int t = threadIdx.x;
    let_next_kernel_start();
    const int64_t tiles = (end - base + kTB - 1) / kTB;
    // the tile's samples (nothing the previous kernel writes)
    float xv = 0.0f, yv = 0.0f;
    auto fetch = [&](int64_t tile) {
        const int64_t b0 = base + tile * kTB;
        if (t < kTB) S.idx[t] = b0 + t < end ? sample_index(b0 + t, n, pa, pc) : -1;
        __syncthreads();
        if (t < kTB * kStopIn) {
            const int i = S.idx[t / kStopIn];
            xv = i >= 0 ? __ldg(X + int64_t(i) * kStopIn + t % kStopIn) : 0.0f;
        } else if (t < kTB * (kStopIn + 1)) {
            const int i = S.idx[t - kTB * kStopIn];
            yv = i >= 0 ? __ldg(Y + i) : 0.0f;
        }
    };
    fetch(blockIdx.x);
    wait_previous_kernel();
    {
        // W2: thread t takes 16 inputs of output row t % 64
        const int o = t & 63, u0 = (t >> 6) * 16;
#pragma unroll
        for (int h = 0; h < 16; h += 8) {
            const uint4 v = __ldcg(reinterpret_cast<const uint4*>(w + kOffW2 + o * kStopH + u0 + h));
            const uint32_t q[4] = {v.x, v.y, v.z, v.w};
            float f[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                __half2 hh;
                memcpy(&hh, &q[i], 4);
                const float2 g = __half22float2(hh);
                f[2 * i] = g.x;
                f[2 * i + 1] = g.y;
            }
            *reinterpret_cast<float4*>(S.w2 + o * kLd + u0 + h) = make_float4(f[0], f[1], f[2], f[3]);
            *reinterpret_cast<float4*>(S.w2 + o * kLd + u0 + h + 4) = make_float4(f[4], f[5], f[6], f[7]);
#pragma unroll
            for (int i = 0; i < 8; ++i) S.w2t[(u0 + h + i) * kLd + o] = f[i];
        }
        for (int i = t; i < kStopH * kStopIn; i += kThreads) S.w1[i] = ld_weight(w + kOffW1 + i);
        if (t < kStopH) {
            S.b1[t] = ld_weight(w + kOffB1 + t);
            S.b2[t] = ld_weight(w + kOffB2 + t);
            S.w3[t] = ld_weight(w + kOffW3 + t);
        }
        if (t < kStopIn) {
            S.mu[t] = __ldcg(norm + t);
            S.isig[t] = 1.0f / __ldcg(norm + kStopIn + t);
        }
    }
    const float b3 = ld_weight(w + kOffB3);
    const int c0 = (t & 15) * 4, r2 = (t >> 4) * 2, r4 = (t >> 4) * 4;  // output tiles: 2x4 of samples, 4x4 of W2
    const int col = t & 63, quarter = t >> 6;
    float g2[4][4] = {};            // W2 gradient, rows r4.., columns c0..
    float gs = 0.0f;                // w3 (quarter 0), b2 (1), b1 (2), b3 and loss (3: threads 192, 193)
    float g1[2] = {0.0f, 0.0f};     // W1 gradient of unit col, inputs quarter and quarter + 4
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        __syncthreads();  // the weights are in place; the last tile's arrays are read
        if (t < kTB * kStopIn) {
            const int f = t % kStopIn;
            S.x[t] = S.idx[t / kStopIn] >= 0 ? (xv - S.mu[f]) * S.isig[f] : 0.0f;
        } else if (t < kTB * (kStopIn + 1)) {
            S.y[t - kTB * kStopIn] = yv;
        }
        __syncthreads();
        // h1 = relu(W1 x + b1): unit col of samples quarter, quarter + 4, ...
        {
            float wr[kStopIn];
#pragma unroll
            for (int f = 0; f < kStopIn; ++f) wr[f] = S.w1[col * kStopIn + f];
            for (int b = quarter; b < kTB; b += 4) {
                float a = S.b1[col];
#pragma unroll
                for (int f = 0; f < kStopIn; ++f) a = fmaf(wr[f], S.x[b * kStopIn + f], a);
                S.h1[b * kLd + col] = fmaxf(a, 0.0f);
            }
        }
        __syncthreads();
        // a2 = W2 h1 + b2
        {
            float o[2][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) o[0][i] = o[1][i] = S.b2[c0 + i];
            tile_2x4(S.h1, S.w2t, r2, c0, o);
#pragma unroll
            for (int r = 0; r < 2; ++r)
                *reinterpret_cast<float4*>(S.a2 + (r2 + r) * kLd + c0) = make_float4(o[r][0], o[r][1], o[r][2], o[r][3]);
        }
        __syncthreads();
        // logit, loss, d loss / d logit, d loss / d a2: 8 lanes per sample, 8 units each
        {
            const int b = t >> 3, u0 = (t & 7) * 8;
            const float4 va = *reinterpret_cast<const float4*>(S.a2 + b * kLd + u0);
            const float4 vb = *reinterpret_cast<const float4*>(S.a2 + b * kLd + u0 + 4);
            float v[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
            float z = 0.0f;
#pragma unroll
            for (int i = 0; i < 8; ++i) z = fmaf(S.w3[u0 + i], fmaxf(v[i], 0.0f), z);
#pragma unroll
            for (int s = 4; s > 0; s >>= 1) z += __shfl_xor_sync(0xffffffffu, z, s);
            z += b3;
            float dz = 0.0f, l = 0.0f;
            if (S.idx[b] >= 0) {
                const float y = S.y[b];
                l = fmaxf(z, 0.0f) - z * y + log1pf(expf(-fabsf(z)));
                dz = (1.0f / (1.0f + expf(-z)) - y) * scale;
            } else {
                // a place past the last sample holds the network's answer to
                // zeros: cleared, so that the sums below add nothing for it
                // (zero times an infinite weight would be NaN)
                const float4 none = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = 0.0f;
#pragma unroll
                for (int i = 0; i < 8; i += 4) {
                    *reinterpret_cast<float4*>(S.a2 + b * kLd + u0 + i) = none;
                    *reinterpret_cast<float4*>(S.h1 + b * kLd + u0 + i) = none;
                }
            }
            if ((t & 7) == 0) {
                S.dz[b] = dz;
                S.ls[b] = l;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = v[i] > 0.0f ? dz * S.w3[u0 + i] : 0.0f;
            *reinterpret_cast<float4*>(S.d2 + b * kLd + u0) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(S.d2 + b * kLd + u0 + 4) = make_float4(v[4], v[5], v[6], v[7]);
        }
        __syncthreads();
        const int64_t next = tile + gridDim.x;
        // d1 = (W2^T d2) masked by a1 > 0
        {
            float o[2][4] = {};
            tile_2x4(S.d2, S.w2, r2, c0, o);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float4 h = *reinterpret_cast<const float4*>(S.h1 + (r2 + r) * kLd + c0);
                *reinterpret_cast<float4*>(S.d1 + (r2 + r) * kLd + c0) =
                    make_float4(h.x > 0.0f ? o[r][0] : 0.0f, h.y > 0.0f ? o[r][1] : 0.0f,
                                h.z > 0.0f ? o[r][2] : 0.0f, h.w > 0.0f ? o[r][3] : 0.0f);
            }
        }
        // W2 gradient: sum over samples of d2 (outer) h1
#pragma unroll 4
        for (int b = 0; b < kTB; ++b) {
            const float4 d = *reinterpret_cast<const float4*>(S.d2 + b * kLd + r4);
            const float4 h = *reinterpret_cast<const float4*>(S.h1 + b * kLd + c0);
            const float p[4] = {d.x, d.y, d.z, d.w}, q[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) g2[i][j] = fmaf(p[i], q[j], g2[i][j]);
        }
        if (quarter == 0) {
            for (int b = 0; b < kTB; ++b) gs = fmaf(S.dz[b], fmaxf(S.a2[b * kLd + col], 0.0f), gs);
        } else if (quarter == 1) {
            for (int b = 0; b < kTB; ++b) gs += S.d2[b * kLd + col];
        } else if (quarter == 3 && col < 2) {
            const float* v = col == 0 ? S.dz : S.ls;
            for (int b = 0; b < kTB; ++b) gs += v[b];
        }
        __syncthreads();
        // W1, b1 gradients
        {
            const bool two = quarter + 4 < kStopIn;
            for (int b = 0; b < kTB; ++b) {
                const float d = S.d1[b * kLd + col];
                g1[0] = fmaf(d, S.x[b * kStopIn + quarter], g1[0]);
                if (two) g1[1] = fmaf(d, S.x[b * kStopIn + quarter + 4], g1[1]);
                if (quarter == 2) gs += d;
            }
        }
        if (next < tiles) fetch(next);
    }
    float* out = part + uint64_t(blockIdx.x) * kPartLd;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4*>(out + kOffW2 + (r4 + i) * kStopH + c0) =
            make_float4(g2[i][0], g2[i][1], g2[i][2], g2[i][3]);
    out[kOffW1 + col * kStopIn + quarter] = g1[0];
    if (quarter + 4 < kStopIn) out[kOffW1 + col * kStopIn + quarter + 4] = g1[1];
    if (quarter == 0) out[kOffW3 + col] = gs;
    if (quarter == 1) out[kOffB2 + col] = gs;
    if (quarter == 2) out[kOffB1 + col] = gs;
    if (quarter == 3 && col == 0) out[kOffB3] = gs;
    if (quarter == 3 && col == 1) out[kStopParams] = gs * scale;
}

// Sum over the blocks' partial rows of column 32 * blockIdx.x + lane: 8
// threads per column, each with every eighth row, then the 8 in order.
// The result is in the block's first warp.
__device__ __forceinline__ float sum_partials(const float* __restrict__ part, int rows) {
    __shared__ float s[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float* p = part + blockIdx.x * 32 + lane;
    float v = 0.0f;
#pragma unroll 8
    for (int r = w; r < rows; r += 8) v += __ldcg(p + uint64_t(r) * kPartLd);
    s[w][lane] = v;
    __syncthreads();
    v = 0.0f;
    if (w == 0)
        for (int i = 0; i < 8; ++i) v += s[i][lane];
    return v;
}

__global__ void __launch_bounds__(256) stop_sum(const float* __restrict__ part, int rows, float* __restrict__ out) {
    const float v = sum_partials(part, rows);
    const int i = blockIdx.x * 32 + threadIdx.x;
    if (threadIdx.x < 32 && i <= kStopParams) out[i] = v;
}

// Adam step on the fp32 master weights from the blocks' partial gradients;
// writes the fp16 working copy and adds the step's loss to *loss.
__global__ void __launch_bounds__(256) stop_adam(float* __restrict__ master, __half* __restrict__ w16,
                                                 const float* __restrict__ part, int rows, float* __restrict__ m1,
                                                 float* __restrict__ m2, float* __restrict__ loss, float lr, float beta1,
                                                 float beta2, float eps, float wd, float c1, float c2) {
    let_next_kernel_start();
    wait_previous_kernel();
    const float sum = sum_partials(part, rows);
    const int i = blockIdx.x * 32 + threadIdx.x;
    if (threadIdx.x >= 32 || i > kStopParams) return;
    if (i == kStopParams) {
        *loss = __ldcg(loss) + sum;
        return;
    }
    const float w = __ldcg(master + i);
    const float g = sum + wd * w;
    const float a = beta1 * __ldcg(m1 + i) + (1.0f - beta1) * g;
    const float b = beta2 * __ldcg(m2 + i) + (1.0f - beta2) * g * g;
    m1[i] = a;
    m2[i] = b;
    const float p = w - lr * (a / c1) / (sqrtf(b / c2) + eps);
    master[i] = p;
    w16[i] = __float2half_rn(p);
}

// Feature sums and sums of squares in fp64, a row of 12 per block (kNormBlocks
// of them: one block alone took 1.0 ms for 200,000 samples), then means and
// standard deviations by the block that the second launch is.
constexpr int kNormBlocks = 128;
__global__ void __launch_bounds__(256) stop_norm(const float* __restrict__ X, int64_t n, double* __restrict__ sums,
                                                 float* __restrict__ norm) {
    __shared__ double s[2 * kStopIn][8];
    double a[kStopIn] = {}, b[kStopIn] = {};
    const bool last = norm != nullptr;
    if (last) {
        if (threadIdx.x < kNormBlocks)
            for (int f = 0; f < kStopIn; ++f) {
                a[f] = sums[threadIdx.x * 2 * kStopIn + f];
                b[f] = sums[threadIdx.x * 2 * kStopIn + kStopIn + f];
            }
    } else {
        for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
            for (int f = 0; f < kStopIn; ++f) {
                const double v = X[i * kStopIn + f];
                a[f] += v;
                b[f] += v * v;
            }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int f = 0; f < kStopIn; ++f) {
        for (int o = 16; o > 0; o >>= 1) {
            a[f] += __shfl_xor_sync(0xffffffffu, a[f], o);
            b[f] += __shfl_xor_sync(0xffffffffu, b[f], o);
        }
        if (lane == 0) {
            s[f][wid] = a[f];
            s[kStopIn + f][wid] = b[f];
        }
    }
    __syncthreads();
    if (threadIdx.x < kStopIn) {
        double sa = 0, sb = 0;
        for (int w = 0; w < int(blockDim.x >> 5); ++w) {
            sa += s[threadIdx.x][w];
            sb += s[kStopIn + threadIdx.x][w];
        }
        if (!last) {
            sums[blockIdx.x * 2 * kStopIn + threadIdx.x] = sa;
            sums[blockIdx.x * 2 * kStopIn + kStopIn + threadIdx.x] = sb;
            return;
        }
        const double mean = sa / double(n);
        const double var = sb / double(n) - mean * mean;
        norm[threadIdx.x] = float(mean);
        norm[kStopIn + threadIdx.x] = float(sqrt(var > 1e-12 ? var : 1e-12));
    }
}

uint64_t splitmix64(uint64_t& s) {
    uint64_t z = (s += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

uint64_t gcd64(uint64_t a, uint64_t b) {
    while (b) {
        const uint64_t t = a % b;
        a = b;
        b = t;
    }
    return a;
}

hnsw_status cuda_err(cudaError_t e, const char* what) {
    return fail(HNSW_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

struct DevBuf {
    void* p = nullptr;
    ~DevBuf() {
        if (p) cudaFree(p);
    }
};

bool bad_device_ptr(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    return !(at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged);
}

size_t smem_bytes() { return sizeof(TrainSmem); }

size_t round256(size_t x) { return (x + 255) & ~size_t(255); }

hnsw_status set_smem() {
    return raise_smem_limit(reinterpret_cast<const void*>(stop_fwd_bwd), smem_bytes(), "stop network");
}

// Blocks for a pass over `samples`: one per tile, up to two per SM.
int fwd_blocks(int64_t samples) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t tiles = (samples + kTB - 1) / kTB;
    return int(tiles < 2 * sms ? tiles : 2 * sms);
}

// Launch with programmatic serialisation (see wait_previous_kernel).
template <class... P, class... A>
cudaError_t launch_next(void (*fn)(P...), int blocks, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(blocks));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

}  // namespace
}  // namespace hnswgb

using namespace hnswgb;

extern "C" hnsw_status hnsw_stop_grad(const float* x, const float* y, int64_t n, const float* norm,
                                      const uint16_t* w_fp16, float* grad_out, float* loss_out, void* stream) {
    if (!x || !y || !norm || !w_fp16 || !grad_out || n < 1) return fail(HNSW_EINVAL, "hnsw_stop_grad: bad argument");
    if (bad_device_ptr(x) || bad_device_ptr(y)) return fail(HNSW_EINVAL, "hnsw_stop_grad: x and y must be device memory");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    hnsw_status st = set_smem();
    if (st != HNSW_OK) return st;
    DevBuf buf;
    // sections start on 256-byte boundaries: [fp16 weights][fp32 grad | loss | norm][partial sums]
    const int blocks = fwd_blocks(n);
    const size_t off_g = round256(size_t(kStopParams) * 2);
    const size_t off_p = off_g + round256((kStopParams + 1 + 2 * kStopIn) * 4);
    const size_t bytes = off_p + size_t(blocks) * kPartLd * 4;
    cudaError_t e = cudaMalloc(&buf.p, bytes);
    if (e != cudaSuccess) return fail(HNSW_ENOMEM, "hnsw_stop_grad: device buffer");
    __half* dw = static_cast<__half*>(buf.p);
    float* dg = reinterpret_cast<float*>(static_cast<char*>(buf.p) + off_g);
    float* dl = dg + kStopParams;
    float* dn = dl + 1;
    float* part = reinterpret_cast<float*>(static_cast<char*>(buf.p) + off_p);
    if ((e = cudaMemcpyAsync(dw, w_fp16, kStopParams * 2, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(dn, norm, 2 * kStopIn * 4, cudaMemcpyHostToDevice, s)) != cudaSuccess)
        return cuda_err(e, "hnsw_stop_grad: copy");
    stop_fwd_bwd<<<blocks, kThreads, smem_bytes(), s>>>(x, y, n, 1, 0, 0, n, dn, dw, part, 1.0f / float(n));
    stop_sum<<<kPartLd / 32, 256, 0, s>>>(part, blocks, dg);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_err(e, "hnsw_stop_grad: launch");
    if ((e = cudaMemcpyAsync(grad_out, dg, kStopParams * 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return cuda_err(e, "hnsw_stop_grad: copy back");
    float l = 0;
    if ((e = cudaMemcpyAsync(&l, dl, 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return cuda_err(e, "hnsw_stop_grad: sync");
    if (loss_out) *loss_out = l;
    return HNSW_OK;
}

extern "C" hnsw_status hnsw_stop_train(const float* x, const float* y, int64_t n, const hnsw_stop_train_params* p,
                                       const uint16_t* w_init, float* norm_out, uint16_t* w_out,
                                       float* loss_per_epoch, void* stream) {
    if (!x || !y || !p || !w_init || !norm_out || !w_out || n < 1)
        return fail(HNSW_EINVAL, "hnsw_stop_train: bad argument");
    if (p->epochs < 1 || p->batch < 128 || p->batch % 128 != 0 || !(p->lr > 0))
        return fail(HNSW_EINVAL, "hnsw_stop_train: epochs >= 1, batch a multiple of 128, lr > 0");
    if (bad_device_ptr(x) || bad_device_ptr(y)) return fail(HNSW_EINVAL, "hnsw_stop_train: x and y must be device memory");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    hnsw_status st = set_smem();
    if (st != HNSW_OK) return st;
    DevBuf buf;
    // sections on 256-byte boundaries: [fp16 weights][master][m1][m2][norm][norm sums][loss per epoch][partial sums]
    const size_t sw = round256(size_t(kStopParams) * 2), sf = round256(size_t(kStopParams) * 4);
    const size_t sn = round256(size_t(kNormBlocks) * 2 * kStopIn * 8), sl = round256(size_t(p->epochs) * 4);
    const int most = fwd_blocks(n < p->batch ? n : p->batch);
    const size_t bytes = sw + 3 * sf + 256 + sn + sl + size_t(most) * kPartLd * 4;
    cudaError_t e = cudaMalloc(&buf.p, bytes);
    if (e != cudaSuccess) return fail(HNSW_ENOMEM, "hnsw_stop_train: device buffer");
    char* c = static_cast<char*>(buf.p);
    __half* dw = reinterpret_cast<__half*>(c);
    float* master = reinterpret_cast<float*>(c + sw);
    float* m1 = reinterpret_cast<float*>(c + sw + sf);
    float* m2 = reinterpret_cast<float*>(c + sw + 2 * sf);
    float* dn = reinterpret_cast<float*>(c + sw + 3 * sf);  // 12 floats
    double* sums = reinterpret_cast<double*>(c + sw + 3 * sf + 256);
    float* dloss = reinterpret_cast<float*>(c + sw + 3 * sf + 256 + sn);  // epochs floats
    float* part = reinterpret_cast<float*>(c + sw + 3 * sf + 256 + sn + sl);
    std::vector<float> mw(kStopParams);
    for (int i = 0; i < kStopParams; ++i) {
        __half_raw r;
        r.x = w_init[i];
        mw[i] = __half2float(__half(r));
    }
    if ((e = cudaMemcpyAsync(dw, w_init, kStopParams * 2, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(master, mw.data(), kStopParams * 4, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemsetAsync(m1, 0, 2 * sf, s)) != cudaSuccess ||
        (e = cudaMemsetAsync(dloss, 0, size_t(p->epochs) * 4, s)) != cudaSuccess)
        return cuda_err(e, "hnsw_stop_train: copy");
    stop_norm<<<kNormBlocks, 256, 0, s>>>(x, n, sums, nullptr);
    stop_norm<<<1, 256, 0, s>>>(x, n, sums, dn);
    const float b1 = p->beta1 > 0 ? p->beta1 : 0.9f, b2 = p->beta2 > 0 ? p->beta2 : 0.999f;
    const float eps = p->eps > 0 ? p->eps : 1e-8f;
    uint64_t rng = p->seed ^ 0x5eed5eedull;
    int step = 0;
    const int64_t steps_per_epoch = (n + p->batch - 1) / p->batch;
    for (int ep = 0; ep < p->epochs; ++ep) {
        // a new affine visiting order of the samples: i -> (a i + c) mod n
        uint64_t a = 1 + splitmix64(rng) % uint64_t(n);
        while (gcd64(a, uint64_t(n)) != 1) a = 1 + (a % uint64_t(n));
        const uint64_t cc = splitmix64(rng) % uint64_t(n);
        for (int64_t k = 0; k < steps_per_epoch; ++k) {
            const int64_t base = k * p->batch;
            const int64_t nb = n - base < p->batch ? n - base : p->batch;
            const int blocks = fwd_blocks(nb);
            e = launch_next(stop_fwd_bwd, blocks, smem_bytes(), s, x, y, n, a, cc, base, base + nb, dn, dw, part,
                            1.0f / float(nb));
            ++step;
            const float c1 = 1.0f - powf(b1, float(step)), c2 = 1.0f - powf(b2, float(step));
            if (e == cudaSuccess)
                e = launch_next(stop_adam, kPartLd / 32, 0, s, master, dw, part, blocks, m1, m2, dloss + ep, p->lr, b1,
                                b2, eps, p->weight_decay, c1, c2);
            if (e != cudaSuccess) return cuda_err(e, "hnsw_stop_train: launch");
        }
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_err(e, "hnsw_stop_train: launch");
    if ((e = cudaMemcpyAsync(w_out, dw, kStopParams * 2, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(norm_out, dn, 2 * kStopIn * 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return cuda_err(e, "hnsw_stop_train: copy back");
    std::vector<float> ls(p->epochs);
    if ((e = cudaMemcpyAsync(ls.data(), dloss, size_t(p->epochs) * 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return cuda_err(e, "hnsw_stop_train: sync");
    if (loss_per_epoch)
        for (int i = 0; i < p->epochs; ++i) loss_per_epoch[i] = ls[i] / float(steps_per_epoch);
    return HNSW_OK;
}

extern "C" hnsw_status hnsw_set_stop_model(hnsw_index* ix, const float* norm, const uint16_t* w_fp16) {
    if (!ix || !norm || !w_fp16) return fail(HNSW_EINVAL, "hnsw_set_stop_model: null argument");
    StopDev h{};
    auto f16 = [&](int i) {
        __half_raw r;
        r.x = w_fp16[i];
        return __half(r);
    };
    for (int i = 0; i < kStopIn; ++i)
        if (!(norm[kStopIn + i] > 0)) return fail(HNSW_EINVAL, "hnsw_set_stop_model: sigma must be > 0");
    // (x - mu) / sigma folded into the first layer
    for (int j = 0; j < kStopH; ++j) {
        double b = double(__half2float(f16(kOffB1 + j)));
        for (int i = 0; i < kStopIn; ++i) {
            const double w = double(__half2float(f16(kOffW1 + j * kStopIn + i))) / double(norm[kStopIn + i]);
            h.w1[j * kStopIn + i] = float(w);
            b -= w * double(norm[i]);
        }
        h.b1[j] = float(b);
    }
    for (int i = 0; i < kStopH; ++i) {
        h.b2[i] = __half2float(f16(kOffB2 + i));
        h.w3[i] = __half2float(f16(kOffW3 + i));
    }
    h.b3 = __half2float(f16(kOffB3));
    for (int u = 0; u < kStopH; ++u)
        for (int l = 0; l < 32; ++l) h.w2p[u * 32 + l] = __halves2half2(f16(kOffW2 + l * kStopH + u), f16(kOffW2 + (l + 32) * kStopH + u));
    if (!ix->d_stop) {
        cudaError_t e = cudaMalloc(&ix->d_stop, sizeof(StopDev));
        if (e != cudaSuccess) {
            ix->d_stop = nullptr;
            return fail(HNSW_ENOMEM, "hnsw_set_stop_model: device buffer");
        }
    }
    cudaError_t e = cudaMemcpy(ix->d_stop, &h, sizeof(StopDev), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_err(e, "hnsw_set_stop_model: copy");
    return HNSW_OK;
}

extern "C" hnsw_status hnsw_clear_stop_model(hnsw_index* ix) {
    if (!ix) return fail(HNSW_EINVAL, "hnsw_clear_stop_model: null index");
    if (ix->d_stop) {
        cudaDeviceSynchronize();
        cudaFree(ix->d_stop);
        ix->d_stop = nullptr;
    }
    return HNSW_OK;
}
