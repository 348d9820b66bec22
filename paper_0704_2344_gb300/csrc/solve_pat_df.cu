// The row-pattern solve kernels of one system in the FP32-pair arithmetic.
#include "solve_pattern.cuh"

namespace fe {
template fe_status dispatch_pat<DFloat>(fe_ctx*, int, SolveParams&);
}  // namespace fe
