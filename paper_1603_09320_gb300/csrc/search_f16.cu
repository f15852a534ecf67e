// search_f16.cu -- the search kernels over fp16 rows.
#include "search_pick.cuh"

namespace hnswgb {

KernelFn search_kernel_f16(const KernelAsk& k) {
    if (k.chunks <= 2) return pick<HNSW_F16, 2, 1, 2, 2>(k);
    if (k.chunks <= 16) return pick<HNSW_F16, 8, 2, HNSW_F16_U, 4>(k);
    if (k.chunks <= 64) return pick<HNSW_F16, 32, 2, 1, 4>(k);
    return nullptr;
}

}  // namespace hnswgb
