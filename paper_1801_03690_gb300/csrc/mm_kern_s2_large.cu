// Single-problem solver kernel for at least 2 x 256 resident threads per SM,
// as one block, in the form for plain FP64 on many rows.
#define MM_BLOCK 512
#define MM_LARGE 1
#include "mm_solver_body.cuh"

namespace mm {
const void* solver_kernel_2_large() { return (const void*)k_solver<2>; }
}  // namespace mm
