// Row passes with the Gram of at most 8 columns of Y' (rowpass_tc.cuh)
#include "rowpass_tc.cuh"

namespace rbo {
TcKernel tc_kernel_g2(bool hc, bool ht) {
  if (ht) return hc ? rowpass_tc_kernel<true, true, 2, false> : rowpass_tc_kernel<false, true, 2, false>;
  return hc ? rowpass_tc_kernel<true, false, 2, false> : rowpass_tc_kernel<false, false, 2, false>;
}
}  // namespace rbo
