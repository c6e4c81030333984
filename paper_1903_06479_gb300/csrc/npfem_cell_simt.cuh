// The persistent SIMT kernel: blocks pull cells from a work counter and solve them alone.
#pragma once

#include "npfem_cell.cuh"

namespace npfem {
namespace {

template <typename T, int MAXT, int MINB, int K>
__global__ void __launch_bounds__(MAXT, MINB) cell_kernel(const __grid_constant__ LaunchArgs<T> a)
{
    unsigned char* smem = smem_dyn;
    CellSolver<T, K> S;
    // first-iterate pass: evaluate only while most cells of the last step were accepted
    const bool eval_first = a.defer && 2ll * (long long)a.defer[2] <= a.total_cells;
    for (;;) {
        const long long item = next_item(a, smem);
        if (item < 0) break;
        if (a.defer && !eval_first) {
            if (threadIdx.x == 0) a.defer[3 + atomicAdd(a.defer, 1u)] = (unsigned int)item;
            continue;
        }
        int gi = 0;
        while (gi + 1 < a.n_groups && item >= a.g[gi + 1].cell_begin) ++gi;
        S.bind(a, a.g[gi], smem);
        if (!S.begin(item - a.g[gi].cell_begin, a.g[gi].stats_off + item - a.g[gi].cell_begin)) continue;
        const bool wants = S.wants_direction();
        if (a.need && wants && threadIdx.x == 0) atomicAdd(a.need, 1u);
        if (a.defer && wants) {
            // the cell needs iterations: the launch that follows solves it from the
            // unchanged state
            if (threadIdx.x == 0) a.defer[3 + atomicAdd(a.defer, 1u)] = (unsigned int)item;
            continue;
        }
        const TopoDev<T>& tp = a.g[gi].topo;
        while (S.wants_direction()) {
            S.first_loop();
            apply_inverse<T, K>(tp, tp.ainv, tp.sp, S.Dv, S.GCv, S.TRIv, S.SPv);  // r = H0 q
            S.second_loop();
            if (!S.descent()) {
                // not a descent direction: drop the history, d = -H~^-1 g
                S.count = 0;
                apply_inverse<T, K>(tp, tp.ainv, tp.sp, S.g, S.GCv, S.TRIv, S.SPv);
                S.negate_direction();
            }
            if (!S.line_search_update()) break;
        }
        S.finish();
    }
    release_counters(a.work, a.total_blocks);
}

}  // namespace
}  // namespace npfem
