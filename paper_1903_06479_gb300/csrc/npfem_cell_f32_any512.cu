// The SIMT kernel, FP32, 512 threads, 1 block per SM, what each mesh has (one translation unit per
// variant: they compile in parallel).
#include "npfem_cell_simt.cuh"

namespace npfem {

const void* cell_kernel_f32_any512() { return reinterpret_cast<const void*>(&cell_kernel<float, 512, 1, kAny>); }

}  // namespace npfem
