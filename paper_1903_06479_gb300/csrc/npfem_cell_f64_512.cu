// The SIMT kernel, FP64, 512 threads, 1 block per SM, sparse solve (one translation unit per
// variant: they compile in parallel).
#include "npfem_cell_simt.cuh"

namespace npfem {

const void* cell_kernel_f64_512() { return reinterpret_cast<const void*>(&cell_kernel<double, 512, 1, kAny>); }

}  // namespace npfem
