// Instantiations of the single-SM tcgen05 GEMM for the data-gradient (A K-major, B MN-major) operand layout.
#include "gemm_tc.cuh"

namespace fl_gemm {
FL_GEMM_INSTANTIATE_SINGLE(, false, true)
}  // namespace fl_gemm
