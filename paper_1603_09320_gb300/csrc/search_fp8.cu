// search_fp8.cu -- the search kernels over fp8 (e4m3) rows.
#include "search_pick.cuh"

namespace hnswgb {

KernelFn search_kernel_fp8(const KernelAsk& k) {
    if (k.chunks <= 8) return pick<HNSW_FP8E4M3, 8, 1, HNSW_FP8_U, 4>(k);
    if (k.chunks <= 32) return pick<HNSW_FP8E4M3, 32, 1, 1, 4>(k);
    return nullptr;
}

}  // namespace hnswgb
