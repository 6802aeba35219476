// Team solver kernel for 256-thread blocks with the inner solve by grid groups,
// compiled in a translation unit of its own so that the library's kernels build
// in parallel.
#include "fct_solver.cuh"

template __global__ void fct_solve_kernel<256, false, 0, true>(const SolveArgs a);
