// Row passes with a general Gram [X Y']^T Y' (rowpass_tc.cuh)
#include "rowpass_tc.cuh"

namespace rbo {
TcKernel tc_kernel_g1(bool hc, bool ht) {
  if (ht) return hc ? rowpass_tc_kernel<true, true, 1, false> : rowpass_tc_kernel<false, true, 1, false>;
  return hc ? rowpass_tc_kernel<true, false, 1, false> : rowpass_tc_kernel<false, false, 1, false>;
}
}  // namespace rbo
