// The cluster kernel for few FP64 cells.
#include "npfem_cell_cluster.cuh"

namespace npfem {

const void* cell_kernel_cl_f64() { return reinterpret_cast<const void*>(&cell_kernel_cl<double>); }

}  // namespace npfem
