// Instantiations of the single-SM tcgen05 GEMM for the forward (A and B K-major) operand layout.
#include "gemm_tc.cuh"

namespace fl_gemm {
FL_GEMM_INSTANTIATE_SINGLE(, false, false)
}  // namespace fl_gemm
