// The row-pattern solve kernels of several systems in the complex64 arithmetic.
#include "solve_pattern.cuh"

namespace fe {
template fe_status launch_pat_jobs<float>(fe_ctx*, int, SolveJob* const*, const int*, int, cudaStream_t, const int*);
}  // namespace fe
