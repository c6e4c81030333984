// The SIMT kernel, FP64, 128 threads, 4 blocks per SM, sparse solve (one translation unit per
// variant: they compile in parallel).
#include "npfem_cell_simt.cuh"

namespace npfem {

const void* cell_kernel_f64_128() { return reinterpret_cast<const void*>(&cell_kernel<double, 128, 4, kAny>); }

}  // namespace npfem
