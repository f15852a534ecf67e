// search_bf16.cu -- the search kernels over bf16 rows.
#include "search_pick.cuh"

namespace hnswgb {

KernelFn search_kernel_bf16(const KernelAsk& k) {
    if (k.chunks <= 2 && !k.check) return pick<HNSW_BF16, 2, 1, 2, 2>(k);
    if (k.chunks <= 16) return pick<HNSW_BF16, 8, 2, HNSW_B16_U, 4, true>(k);
    if (k.chunks <= 64) return pick<HNSW_BF16, 32, 2, 1, 4>(k);
    return nullptr;
}

}  // namespace hnswgb
