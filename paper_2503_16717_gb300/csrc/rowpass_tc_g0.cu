// Row passes without a Gram: update, triangular solve, sketch (rowpass_tc.cuh)
#include "rowpass_tc.cuh"

namespace rbo {
TcKernel tc_kernel_g0(bool hc, bool ht, bool sk) {
  if (sk) return ht ? nullptr : (hc ? rowpass_tc_kernel<true, false, 0, true> : rowpass_tc_kernel<false, false, 0, true>);
  if (ht) return hc ? rowpass_tc_kernel<true, true, 0, false> : rowpass_tc_kernel<false, true, 0, false>;
  return hc ? rowpass_tc_kernel<true, false, 0, false> : rowpass_tc_kernel<false, false, 0, false>;
}
}  // namespace rbo
