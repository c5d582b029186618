// Row passes with the Gram of at most 8 columns of Y' (rowpass_tc.cuh)
#include "rowpass_tc.cuh"

namespace rbo {
TcKernel tc_kernel_g2(bool hc, int tri) {
  if (hc) return tri ? nullptr : rowpass_tc_kernel<true, 0, 2, false>;
  if (tri == 2) return nullptr;  // (the inverse is for wider panels)
  if (tri) return rowpass_tc_kernel<false, 1, 2, false>;
  return rowpass_tc_kernel<false, 0, 2, false>;
}
}  // namespace rbo
