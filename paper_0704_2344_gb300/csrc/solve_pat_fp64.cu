// The row-pattern solve kernels of one system in the complex128 arithmetic.
#include "solve_pattern.cuh"

namespace fe {
template fe_status dispatch_pat<double>(fe_ctx*, int, SolveParams&);
}  // namespace fe
