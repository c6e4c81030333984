// The tensor-core kernel with 16 result columns per cluster.
#include "npfem_cell_tc.cuh"

namespace npfem {

const void* cell_kernel_tc16() { return reinterpret_cast<const void*>(&cell_kernel_tc<float, 16, kDense>); }

}  // namespace npfem
