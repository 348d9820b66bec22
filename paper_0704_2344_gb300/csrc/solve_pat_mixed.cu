// The row-pattern solve kernels of one system in the complex64 arithmetic.
#include "solve_pattern.cuh"

namespace fe {
template fe_status dispatch_pat<float>(fe_ctx*, int, SolveParams&);
}  // namespace fe
