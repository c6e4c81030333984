// The tensor-core kernel with 32 result columns per cluster for meshes with beta_D > 0
// (dense M~^-1: the call of the sparse solve made the rest of it 5 to 8 % slower).
#include "npfem_cell_tc.cuh"

namespace npfem {

const void* cell_kernel_tc32_damped() { return reinterpret_cast<const void*>(&cell_kernel_tc<float, 32, kDenseDamped>); }

}  // namespace npfem
