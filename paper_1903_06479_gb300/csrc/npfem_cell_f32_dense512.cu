// The SIMT kernel, FP32, 512 threads, 1 block per SM, dense inverse (one translation unit per
// variant: they compile in parallel).
#include "npfem_cell_simt.cuh"

namespace npfem {

const void* cell_kernel_f32_dense512() { return reinterpret_cast<const void*>(&cell_kernel<float, 512, 1, kDense>); }

}  // namespace npfem
