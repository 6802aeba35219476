// Team solver kernels for 256-thread blocks with the inner solve by grid groups
// (for batches and servers, and in the deep-gather variant for one transform),
// compiled in a translation unit of their own so that the library's kernels build
// in parallel.
#include "fct_solver.cuh"

template __global__ void fct_solve_kernel<256, false, 0, true>(const SolveArgs a);
template __global__ void fct_solve_kernel<256, false, 1, true>(const SolveArgs a);
