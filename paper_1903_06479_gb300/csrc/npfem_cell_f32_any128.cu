// The SIMT kernel, FP32, 128 threads, 4 blocks per SM, what each mesh has (one translation unit per
// variant: they compile in parallel).
#include "npfem_cell_simt.cuh"

namespace npfem {

const void* cell_kernel_f32_any128() { return reinterpret_cast<const void*>(&cell_kernel<float, 128, 4, kAny>); }

}  // namespace npfem
