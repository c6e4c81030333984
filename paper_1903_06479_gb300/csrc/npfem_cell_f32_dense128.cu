// The SIMT kernel, FP32, 128 threads, 4 blocks per SM, dense inverse (one translation unit per
// variant: they compile in parallel).
#include "npfem_cell_simt.cuh"

namespace npfem {

const void* cell_kernel_f32_dense128() { return reinterpret_cast<const void*>(&cell_kernel<float, 128, 4, kDense>); }

}  // namespace npfem
