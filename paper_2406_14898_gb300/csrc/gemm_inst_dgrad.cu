// Instantiations of the CTA-pair tcgen05 GEMM for the data-gradient (A K-major, B MN-major) operand layout.
#include "gemm_tc.cuh"

namespace fl_gemm {
FL_GEMM_INSTANTIATE_PAIR(, false, true)
}  // namespace fl_gemm
