// On-chip solves whose iterate is float64 (resident_solve.cuh).
#include "resident_solve.cuh"

namespace pdhg {
template const void* res_solve_kernel<double>(int, bool);
template cudaError_t launch_res_solve<double>(const ResSolve<double>&, int, int, size_t, bool, cudaStream_t);
}  // namespace pdhg
