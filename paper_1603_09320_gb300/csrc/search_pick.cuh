// search_pick.cuh -- choice of a search kernel's instantiation for one row
// format; each storage type's translation unit (search_f32.cu, ...) lists its
// formats.
#pragma once

#include "search_kernel.cuh"
#include "search_team.cuh"

namespace hnswgb {

// Rows of up to TEAM * CPL chunks: U rows in flight per team of lanes in the
// warp-per-query kernel, UT in the block-per-query one; CHECKED: the
// bounds-checked build exists for this format.
template <int ST, int TEAM, int CPL, int U, bool CHECKED, bool FULL>
KernelFn pick_full(const KernelAsk& k) {
    if (k.check) {
        if constexpr (CHECKED)
            return k.wide ? hnsw_search_kernel<ST, TEAM, CPL, U, FULL, false, true, true>
                          : hnsw_search_kernel<ST, TEAM, CPL, U, FULL, false, false, true>;
        return nullptr;
    }
    if (k.stop)
        return k.wide ? hnsw_search_kernel<ST, TEAM, CPL, U, FULL, true, true>
                      : hnsw_search_kernel<ST, TEAM, CPL, U, FULL, true, false>;
    return k.wide ? hnsw_search_kernel<ST, TEAM, CPL, U, FULL, false, true>
                  : hnsw_search_kernel<ST, TEAM, CPL, U, FULL, false, false>;
}

template <int ST, int TEAM, int CPL, int U, int UT, bool CHECKED = false>
KernelFn pick(const KernelAsk& k) {
    if (k.team_r)
        return k.team_r == 2   ? hnsw_team_kernel<ST, TEAM, CPL, UT, 2>
               : k.team_r == 8 ? hnsw_team_kernel<ST, TEAM, CPL, UT, 8>
                               : hnsw_team_kernel<ST, TEAM, CPL, UT, 16>;
    return k.chunks == uint32_t(TEAM * CPL) ? pick_full<ST, TEAM, CPL, U, CHECKED, true>(k)
                                            : pick_full<ST, TEAM, CPL, U, CHECKED, false>(k);
}

}  // namespace hnswgb
