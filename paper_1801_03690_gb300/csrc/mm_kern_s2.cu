// Single-problem solver kernel for at least 2 x 256 resident threads per SM,
// as one block.
#define MM_BLOCK 512
#include "mm_solver_body.cuh"

namespace mm {
const void* solver_kernel_2() { return (const void*)k_solver<2>; }
}  // namespace mm
