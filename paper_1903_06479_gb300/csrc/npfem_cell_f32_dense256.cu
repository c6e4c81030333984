// The SIMT kernel, FP32, 256 threads, 2 blocks per SM, dense inverse (one translation unit per
// variant: they compile in parallel).
#include "npfem_cell_simt.cuh"

namespace npfem {

const void* cell_kernel_f32_dense256() { return reinterpret_cast<const void*>(&cell_kernel<float, 256, 2, kDense>); }

}  // namespace npfem
