// The cluster kernel for few FP64 cells: the blocks of a cluster solve one cell together
// (Team in npfem_cell.cuh), for launches with fewer cells than SMs, where a block per cell
// would leave the other SMs idle.  One block is bound by its SM's FP64 pipe (about 1650 FP64
// instructions per triangle and evaluation); eight share them, and what is left is the
// latency of one triangle's chain (one 258-vertex cell, four steps: 10.9 ms by one block of
// 512 threads, 6.18 by eight of 512, 4.64 by eight of 128, which do not run the reductions
// on warps without data).  FP32 stays at a block per cell: with eight blocks of 512 threads and
// the sparse solve (a cluster barrier per level) one 642-vertex cell took 1.35 ms for eight
// steps, by one block with the dense inverse 1.31; blocks of 128 threads, or a cluster that
// only shares the dense contraction, were not tried.  Clusters take the cells in turn.
#pragma once

#include "npfem_cell.cuh"

namespace npfem {
namespace {

template <typename T>
__global__ void __launch_bounds__(512, 1) cell_kernel_cl(const __grid_constant__ LaunchArgs<T> a)
{
    unsigned char* smem = smem_dyn;
    CellShared<T>* sh = cell_shared<T>(smem);
    uint32_t rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int C = a.p.cluster;
    if (threadIdx.x == 0) {
        sh->cl_size = C;
        sh->cl_rank = (int)rank;
        sh->cl_par = 0;
    }
    __syncthreads();
    cluster_barrier();
    CellSolver<T, kDense, true> S;
    for (long long item = blockIdx.x / C; item < a.total_cells; item += gridDim.x / C) {
        int gi = 0;
        while (gi + 1 < a.n_groups && item >= a.g[gi + 1].cell_begin) ++gi;
        S.bind(a, a.g[gi], smem);
        S.begin(item - a.g[gi].cell_begin, a.g[gi].stats_off + item - a.g[gi].cell_begin);
        const TopoDev<T>& tp = a.g[gi].topo;
        while (S.wants_direction()) {
            S.first_loop();
            solve_sparse<T, true>(tp.spc, S.tm, tp.n, S.Dv, S.GCv, S.SPv);  // r = H0 q
            S.second_loop();
            if (!S.descent()) {
                // not a descent direction: drop the history, d = -H~^-1 g
                S.count = 0;
                S.first_loop();
                solve_sparse<T, true>(tp.spc, S.tm, tp.n, S.Dv, S.GCv, S.SPv);
                S.negate_direction();
            }
            if (!S.line_search_update()) break;
        }
        S.finish();
        // no block writes the next cell into shared memory another still reads
        cluster_barrier();
    }
}

}  // namespace
}  // namespace npfem
