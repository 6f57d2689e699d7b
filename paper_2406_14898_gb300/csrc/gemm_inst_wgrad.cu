// Instantiations of the CTA-pair tcgen05 GEMM for the weight-gradient (A and B MN-major) operand layout.
#include "gemm_tc.cuh"

namespace fl_gemm {
FL_GEMM_INSTANTIATE_PAIR(, true, true)
FL_GEMM_INSTANTIATE_WGRAD()
}  // namespace fl_gemm
