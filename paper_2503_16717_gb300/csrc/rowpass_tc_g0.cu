// Row passes without a Gram: update, triangular solve, sketch (rowpass_tc.cuh)
#include "rowpass_tc.cuh"

namespace rbo {
TcKernel tc_kernel_g0(bool hc, int tri, bool sk) {
  if (sk) return tri ? nullptr : (hc ? rowpass_tc_kernel<true, 0, 0, true> : rowpass_tc_kernel<false, 0, 0, true>);
  if (hc) return tri ? nullptr : rowpass_tc_kernel<true, 0, 0, false>;
  if (tri) return tri == 2 ? rowpass_tc_kernel<false, 2, 0, false> : rowpass_tc_kernel<false, 1, 0, false>;
  return nullptr;
}
}  // namespace rbo
