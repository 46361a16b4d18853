// Single-problem solver kernel for at least 4 x 256 resident threads per SM,
// as one block.
#define MM_BLOCK 1024
#include "mm_solver_body.cuh"

namespace mm {
const void* solver_kernel_4() { return (const void*)k_solver<4>; }
}  // namespace mm
