// Tensor copies of 16-row boxes of a column-major float64 array (the 128-byte swizzled
// tile layout of tc_tile.cuh and of the digit Gram in ozaki.cu).
#pragma once

#include <cuda.h>

#include "device_common.cuh"

namespace rbo {

// 2-D tensor map of a column-major float64 array (n rows, cols columns, leading
// dimension ld even, base 16-byte aligned): boxes of 16 rows x cols columns with the
// 128-byte swizzle, out-of-range rows read as zero.
int make_tensor_map(CUtensorMap* m, const double* base, int64_t n, int cols, int64_t ld);

// box starting at row x0 into shared memory (1024-byte aligned), completion on `bar`
__device__ __forceinline__ void tma_load_rows(void* dst, const CUtensorMap* tm, int x0, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(smem_u32(dst)),
      "l"(tm), "r"(x0), "r"(0), "r"(smem_u32(bar))
      : "memory");
}

}  // namespace rbo
