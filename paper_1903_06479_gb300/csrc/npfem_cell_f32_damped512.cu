// The SIMT kernel, FP32, 512 threads, 1 block per SM, dense inverses, beta_D > 0 (one translation unit per
// variant: they compile in parallel).
#include "npfem_cell_simt.cuh"

namespace npfem {

const void* cell_kernel_f32_damped512() { return reinterpret_cast<const void*>(&cell_kernel<float, 512, 1, kDenseDamped>); }

}  // namespace npfem
