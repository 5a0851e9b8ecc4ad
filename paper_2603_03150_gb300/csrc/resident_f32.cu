// On-chip solves whose iterate is float32 (resident_solve.cuh).
#include "resident_solve.cuh"

namespace pdhg {
template const void* res_solve_kernel<float>(int, bool);
template cudaError_t launch_res_solve<float>(const ResSolve<float>&, int, int, size_t, bool, cudaStream_t);
}  // namespace pdhg
