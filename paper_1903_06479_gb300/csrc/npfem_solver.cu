// Launches of the solver kernels: the variant of a launch (scalar type, block size), its
// shared memory, occupancy and cluster attributes.
#include <cuda_runtime.h>

#include "npfem_internal.h"

namespace npfem {

// npfem_cell_*.cu
const void* cell_kernel_f32_dense512();
const void* cell_kernel_f32_dense256();
const void* cell_kernel_f32_dense128();
const void* cell_kernel_f32_damped512();
const void* cell_kernel_f32_damped256();
const void* cell_kernel_f32_damped128();
const void* cell_kernel_f32_any512();
const void* cell_kernel_f32_any256();
const void* cell_kernel_f32_any128();
const void* cell_kernel_f64_512();
const void* cell_kernel_f64_128();
const void* cell_kernel_cl_f64();
const void* cell_kernel_tc16();
const void* cell_kernel_tc32();
const void* cell_kernel_tc32_damped();

namespace {

// The narrowest variant that has what every topology of the launch applies.  An evaluation
// applies nothing, a first-iterate pass (defer) M~^-1 at most.
enum { kOfDense, kOfDamped, kOfAny };
int variant(const LaunchArgs<float>& a)
{
    int v = kOfDense;
    for (int g = 0; g < a.n_groups && a.p.mode == 0; ++g) {
        const TopoDev<float>& tp = a.g[g].topo;
        if ((!tp.ainv && !a.defer) || (tp.l_ptr && !tp.minv)) return kOfAny;
        if (tp.l_ptr) v = kOfDamped;
    }
    return v;
}

const void* simt_kernel(const LaunchArgs<double>&, int block)
{
    return block == 512 ? cell_kernel_f64_512() : (block == 128 ? cell_kernel_f64_128() : nullptr);
}

const void* simt_kernel(const LaunchArgs<float>& a, int block)
{
    using Get = const void* (*)();
    static const Get by[3][3] = {{cell_kernel_f32_dense512, cell_kernel_f32_dense256, cell_kernel_f32_dense128},
                                 {cell_kernel_f32_damped512, cell_kernel_f32_damped256, cell_kernel_f32_damped128},
                                 {cell_kernel_f32_any512, cell_kernel_f32_any256, cell_kernel_f32_any128}};
    const int b = block == 512 ? 0 : (block == 256 ? 1 : (block == 128 ? 2 : -1));
    return b < 0 ? nullptr : by[variant(a)][b]();
}

const void* tc_kernel(int cluster, bool damped)
{
    if (cluster * 3 <= 16) return damped ? nullptr : cell_kernel_tc16();
    return damped ? cell_kernel_tc32_damped() : cell_kernel_tc32();
}

cudaLaunchConfig_t tc_config(int cluster, int block, int smem, int grid, cudaStream_t s, cudaLaunchAttribute* attr)
{
    cudaLaunchConfig_t cfg = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(block);
    cfg.gridDim = dim3(grid);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

cudaError_t allow_smem(const void* k, int limit)
{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
}

template <typename T>
cudaError_t allow_cells_smem(const LaunchArgs<T>& a, int block, int limit)
{
    const void* k = simt_kernel(a, block);
    return k ? allow_smem(k, limit) : cudaErrorInvalidValue;
}

template <typename T>
cudaError_t cells_per_sm(const LaunchArgs<T>& a, int block, int smem, int limit, int* n)
{
    const void* k = simt_kernel(a, block);
    if (!k) return cudaErrorInvalidValue;
    cudaError_t e = allow_smem(k, limit);
    return e == cudaSuccess ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k, block, smem) : e;
}

template <typename T>
cudaError_t launch_cells(const LaunchArgs<T>& a, int grid, int block, int smem, cudaStream_t s)
{
    const void* k = simt_kernel(a, block);
    if (!k) return cudaErrorInvalidValue;
    void* args[1] = {const_cast<LaunchArgs<T>*>(&a)};
    const cudaError_t e = cudaLaunchKernel(k, dim3(grid), dim3(block), args, smem, s);
    if (e == cudaSuccess) count_launch();
    return e;
}

cudaError_t query_cells_cl(int cluster, int block, int smem, int limit, int* max_clusters)
{
    const void* k = cell_kernel_cl_f64();
    cudaError_t e = allow_smem(k, limit);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = tc_config(cluster, block, smem, cluster, nullptr, attr);
    return cudaOccupancyMaxActiveClusters(max_clusters, k, &cfg);
}

cudaError_t launch_cells_cl(const LaunchArgs<double>& a, int cluster, int clusters, int block, int smem, cudaStream_t s)
{
    const void* k = cell_kernel_cl_f64();
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = tc_config(cluster, block, smem, cluster * clusters, s, attr);
    void* args[1] = {const_cast<LaunchArgs<double>*>(&a)};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, k, args);
    if (e == cudaSuccess) count_launch();
    return e;
}

cudaError_t query_cells_tc(int cluster, bool damped, int block, int smem, int limit, int* max_clusters)
{
    const void* k = tc_kernel(cluster, damped);
    if (!k) return cudaErrorInvalidValue;
    cudaError_t e = allow_smem(k, limit);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = tc_config(cluster, block, smem, cluster, nullptr, attr);
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
    if (e != cudaSuccess) return e;
    if (n < 1) return cudaErrorInvalidConfiguration;
    *max_clusters = n;
    return cudaSuccess;
}

// Cluster launch of the tensor-core kernel for one mesh group.
cudaError_t launch_cells_tc(const LaunchArgs<float>& a, int cluster, int block, int smem, int grid, cudaStream_t s)
{
    const void* k = tc_kernel(cluster, a.g[0].topo.l_ptr != nullptr);
    if (!k) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = tc_config(cluster, block, smem, grid, s, attr);
    void* args[1] = {const_cast<LaunchArgs<float>*>(&a)};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, k, args);
    if (e == cudaSuccess) count_launch();
    return e;
}

template cudaError_t launch_cells<float>(const LaunchArgs<float>&, int, int, int, cudaStream_t);
template cudaError_t launch_cells<double>(const LaunchArgs<double>&, int, int, int, cudaStream_t);
template cudaError_t allow_cells_smem<float>(const LaunchArgs<float>&, int, int);
template cudaError_t cells_per_sm<float>(const LaunchArgs<float>&, int, int, int, int*);
template cudaError_t cells_per_sm<double>(const LaunchArgs<double>&, int, int, int, int*);

}  // namespace npfem
