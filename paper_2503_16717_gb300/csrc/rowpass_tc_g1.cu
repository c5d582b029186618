// Row passes with a general Gram [X Y']^T Y' (rowpass_tc.cuh)
#include "rowpass_tc.cuh"

namespace rbo {
TcKernel tc_kernel_g1(bool hc, int tri) {
  if (hc) return tri ? rowpass_tc_kernel<true, 1, 1, false> : nullptr;
  if (tri) return tri == 2 ? rowpass_tc_kernel<false, 2, 1, false> : rowpass_tc_kernel<false, 1, 1, false>;
  return rowpass_tc_kernel<false, 0, 1, false>;
}
TcKernel tc_kernel_g3() { return rowpass_tc_kernel<true, 0, 3, false>; }
TcKernel tc_kernel_g4() { return rowpass_tc_kernel<false, 0, 4, false>; }
}  // namespace rbo
