// Single-problem solver kernel for at least 3 x 256 resident threads per SM,
// as one block.
#define MM_BLOCK 768
#include "mm_solver_body.cuh"

namespace mm {
const void* solver_kernel_3() { return (const void*)k_solver<3>; }
}  // namespace mm
