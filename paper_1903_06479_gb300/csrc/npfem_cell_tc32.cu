// The tensor-core kernel with 32 result columns per cluster.
#include "npfem_cell_tc.cuh"

namespace npfem {

const void* cell_kernel_tc32() { return reinterpret_cast<const void*>(&cell_kernel_tc<float, 32, kDense>); }

}  // namespace npfem
