// search_f32.cu -- the search kernels over fp32 rows.
#include "search_pick.cuh"

namespace hnswgb {

KernelFn search_kernel_f32(const KernelAsk& k) {
    if (k.chunks <= 2 && !k.check) return pick<HNSW_F32, 2, 1, 2, 2>(k);
    if (k.chunks <= 8) return pick<HNSW_F32, 8, 1, 8, 4, true>(k);
    if (k.chunks <= 32) return pick<HNSW_F32, 8, 4, HNSW_F32_U, 4, true>(k);
    if (k.chunks <= 128) return pick<HNSW_F32, 32, 4, 1, 4>(k);
    return nullptr;
}

}  // namespace hnswgb
