// Instantiations of the single-SM tcgen05 GEMM for the weight-gradient (A and B MN-major) operand layout.
#include "gemm_tc.cuh"

namespace fl_gemm {
FL_GEMM_INSTANTIATE_SINGLE(, true, true)
}  // namespace fl_gemm
