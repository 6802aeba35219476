// Team solver kernels for 128-thread blocks (with and without staged entry
// values), compiled in a translation unit of their own so that the library's
// kernels build in parallel.
#include "fct_solver.cuh"

template __global__ void fct_solve_kernel<128, false, 0, false>(const SolveArgs a);
template __global__ void fct_solve_kernel<128, true, 0, false>(const SolveArgs a);
