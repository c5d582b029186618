// CSR sparse kernels of the matrix-powers kernel (Section 4) and the small vector
// kernels of the GMRES driver.
//
// SpMV: rows of up to ~12 entries on average (stencils) go to a kernel in which each
// block stages the entries of 256 consecutive rows in shared memory and every thread
// runs its own row; denser rows use a group of LPR = 8 or 32 lanes per row that read
// consecutive entries and combine with shuffles in a fixed order.
// Every sum has a fixed order, so the result is deterministic.  The optional
// diagonal scaling D of the right Jacobi preconditioner (A D x) is applied to the
// gathered x entries; the optional shift terms of the Newton and Chebyshev bases
// are added to each output row.
#include <algorithm>
#include <vector>

#include "device_common.cuh"

namespace rbo {

// (A x)_r + a u_r + b uprev_r, in the order of the separate shift pass
__device__ __forceinline__ double shifted(double s, const SpmvShift& sh, int64_t r) {
  if (!sh.u) return s;
  double v = fma(sh.a, sh.u[r], s);
  if (sh.uprev) v = fma(sh.b, sh.uprev[r], v);
  return v;
}

// Entries with a column index outside [0, n), or rows whose pointers leave [0, nnz],
// are skipped and reported through the status word (RBO_ERR_ARG) instead of being
// dereferenced.
template <int LPR>
__global__ void __launch_bounds__(256) spmv_kernel(int64_t n, int64_t nnz,
                                                   const int32_t* __restrict__ rowptr,
                                                   const int32_t* __restrict__ col,
                                                   const double* __restrict__ val,
                                                   const double* __restrict__ dscale,
                                                   const double* __restrict__ x,
                                                   const double* __restrict__ bvec,
                                                   double* __restrict__ y, DevStatus* status,
                                                   SpmvShift sh) {
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t row = gid / LPR;
  const int sub = (int)(gid % LPR);
  double s = 0.0;
  if (row < n) {
    int beg = __ldg(rowptr + row), end = __ldg(rowptr + row + 1);
    if (beg < 0 || end < beg || (int64_t)end > nnz) {
      if (status && sub == 0) set_error(status, RBO_ERR_ARG, 11);
      end = beg;
    }
      for (int j = beg + sub; j < end; j += LPR) {
        const int cj = __ldg(col + j);
        if (cj < 0 || (int64_t)cj >= n) {
          if (status) set_error(status, RBO_ERR_ARG, 12);
          continue;
        }
        const double xv = dscale ? __ldg(dscale + cj) * __ldg(x + cj) : __ldg(x + cj);
        s = fma(__ldg(val + j), xv, s);
      }
  }
#pragma unroll
  for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, LPR);
  if (row < n && sub == 0) y[row] = bvec ? (bvec[row] - s) : shifted(s, sh, row);
}


// Short rows: a block takes 256 consecutive rows, whose indices and values are two
// contiguous pieces of the CSR arrays; the bulk-copy engine brings them into shared memory
// (no load instructions and no registers for the bytes in flight, which bound an earlier
// form that staged 32 rows per warp with plain loads), then every thread walks its own row,
// the x gathers of 8 entries in flight.  Two interleaved chains per row (even and odd
// entries) added at the end, a fixed order; no cross-lane float64 reduction.  Arrays that are
// not 16-byte aligned are staged with plain loads.  SCALE is a template argument because the
// float64 pipe (2 operations per SM and cycle) bounds the kernel: a multiplication by a scale
// that is not there would be half of its work.  32 rows a warp staged with plain loads -> here:
// 7-point 100^3 39 -> 24 us, 5-point 2048^2 111 -> 64 us (78 % of the copy rate); one row per
// thread straight from global memory 45 and 139 us.  8 blocks per SM (32 registers): the solve of
// 60 iterations at 2048^2 takes 41.2 ms, with 6 blocks 42.4.
// Blocks with more entries than the staging holds (`cap`) stage them piece by piece.  There a
// row of more than SPL_WARP entries is summed by its warp and one of more than SPL_BLOCK by
// the block, so that no thread walks a long row alone while the others wait (10^6 rows, one of
// 100000 entries: 5.0 ms staged per warp, 10 ms walked by its thread, 0.2 ms here; rows of 20 and
// of 2 entries, half each: 165 us walked from global memory, 100 us in pieces).
constexpr int SPR = 256;         // rows (threads) per block
constexpr int SPL_WARP = 128;    // about where a thread's chain of gathers takes as long as the
                                 // warp's turn and its reduction
constexpr int SPL_BLOCK = 4096;  // 16 turns of a warp; 2 of the block, whose reduction has barriers
struct SpmvArgs {
  int64_t n, nnz;
  const int32_t* rowptr;
  const int32_t* col;
  const double* val;
  const double* dscale;
  const double* x;
  const double* bvec;
  double* y;
  DevStatus* status;
  SpmvShift sh;
  uint32_t ncol;  // columns that a 32-bit index can name: min(n, 2^31)
  int cap, bulk;  // entries that the staging holds; arrays are aligned for bulk copies
};
// entries cp[0..len), vp[0..len) added to the two chains; bad: a column outside the matrix.
// Whole warp: the lanes leave the products of a turn together, after the warp's longest row,
// since a float64 operation takes its pipe for 16 cycles for one lane as for 32, and when its
// predicate is off in all of them (5 entries a row at 2048^2: 83 -> 64 us).
template <bool SCALE, int U>
__device__ __forceinline__ void spmv_walk(const SpmvArgs& A, const int32_t* cp, const double* vp, int len, double& s0,
                                          double& s1, bool& bad) {
  const int longest = __reduce_max_sync(0xffffffffu, len);
  for (int e = 0; e < longest; e += U) {
    const int k = len - e, kw = longest - e;  // entries left
    int c[U];
    double xv[U], dv[SCALE ? U : 1];
#pragma unroll
    for (int j = 0; j < U; ++j) c[j] = j < k ? cp[e + j] : -1;
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const bool ok = (uint32_t)c[j] < A.ncol;
      bad = bad || (j < k && !ok);
      xv[j] = 0.0;
      if (SCALE) dv[j] = 0.0;
      if (ok) {
        xv[j] = __ldg(A.x + c[j]);
        if (SCALE) dv[j] = __ldg(A.dscale + c[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      if (j >= kw) break;
      const double t = SCALE ? dv[j] * xv[j] : xv[j], v = j < k ? vp[e + j] : 0.0;
      if (j & 1) s1 = fma(v, t, s1);
      else s0 = fma(v, t, s0);
    }
  }
}

// row pointers of row r, whose block's entries are e0 .. e1 - 1 (range: a part of the arrays); a
// row that is not part of them is reported and left empty
__device__ __forceinline__ void spmv_row(const SpmvArgs& A, int64_t r, int e0, int e1, bool range, int& beg, int& end) {
  beg = end = 0;
  if (r >= A.n) return;
  beg = __ldg(A.rowptr + r);
  end = __ldg(A.rowptr + r + 1);
  if (range ? (beg < e0 || end < beg || end > e1) : (beg < 0 || end < beg || (int64_t)end > A.nnz)) {
    if (A.status) set_error(A.status, RBO_ERR_ARG, 11);
    end = beg;
  }
}
__device__ __forceinline__ void spmv_store(const SpmvArgs& A, int64_t r, double s, bool bad) {
  if (bad && A.status) set_error(A.status, RBO_ERR_ARG, 12);
  if (r < A.n) A.y[r] = A.bvec ? (A.bvec[r] - s) : shifted(s, A.sh, r);
}

// Sum of this thread's row where it is a long one, else 0: rows of more than SPL_WARP entries by
// their warp, of more than SPL_BLOCK by the block.  Whole block.
template <bool SCALE>
__device__ __noinline__ double spmv_long_rows(const SpmvArgs& A, int64_t r0, int beg, int len) {
  __shared__ double s_red[32];
  __shared__ unsigned s_long[SPR / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double s0 = 0.0;
  bool bad = false;
  // part of a long row: entries id, id + step, ..
  auto part = [&](int from, int cnt, int id, int step) {
    double t = 0.0;
    for (int64_t e = id; e < cnt; e += 4 * (int64_t)step) {
      double p[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t q = e + u * (int64_t)step;
        p[u] = 0.0;
        if (q < cnt) {
          const int cj = __ldg(A.col + from + q);
          const bool ok = (uint32_t)cj < A.ncol;
          bad = bad || !ok;
          if (ok) p[u] = __ldg(A.val + from + q) * (SCALE ? __ldg(A.dscale + cj) * __ldg(A.x + cj) : __ldg(A.x + cj));
        }
      }
      t += (p[0] + p[1]) + (p[2] + p[3]);
    }
    return t;
  };
  for (unsigned m = __ballot_sync(0xffffffffu, len > SPL_WARP && len <= SPL_BLOCK); m; m &= m - 1u) {
    const int l = __ffs((int)m) - 1;
    const double t = warp_sum(part(__shfl_sync(0xffffffffu, beg, l), __shfl_sync(0xffffffffu, len, l), lane, 32));
    if (lane == l) s0 = t;
  }
  const unsigned lb = __ballot_sync(0xffffffffu, len > SPL_BLOCK);
  if (lane == 0) s_long[warp] = lb;
  __syncthreads();
  for (int w = 0; w < SPR / 32; ++w)
    for (unsigned m = s_long[w]; m; m &= m - 1u) {
      const int t = 32 * w + __ffs((int)m) - 1, from = __ldg(A.rowptr + r0 + t);
      const double v = block_sum(part(from, __ldg(A.rowptr + r0 + t + 1) - from, tid, SPR), s_red);
      if (tid == t) s0 = v;
    }
  if (bad && A.status) set_error(A.status, RBO_ERR_ARG, 12);
  return s0;
}

// A block whose entries do not fit the staging at once, or whose row pointers are out of order.
// Apart from the kernel, whose registers it would take.
template <bool SCALE>
__device__ __noinline__ void spmv_pieces(const SpmvArgs& A, double* sval, int32_t* scol) {
  const int tid = threadIdx.x, cap = A.cap;
  const int64_t r0 = blockIdx.x * (int64_t)SPR, r = r0 + tid;
  const int e0 = __ldg(A.rowptr + r0), e1 = __ldg(A.rowptr + (r0 + SPR < A.n ? r0 + SPR : A.n));
  const bool range = e0 >= 0 && e1 >= e0 && (int64_t)e1 <= A.nnz;
  int beg, end;
  spmv_row(A, r, e0, e1, range, beg, end);
  const int len = end - beg;
  const bool lng = len > SPL_WARP;
  double s0 = 0.0, s1 = 0.0;
  bool bad = false;
  if (!range) {  // the rows that lie in the arrays
    spmv_walk<SCALE, SCALE ? 2 : 4>(A, A.col + beg, A.val + beg, len, s0, s1, bad);
    spmv_store(A, r, s0 + s1, bad);
    return;
  }
  for (int64_t k0 = e0; k0 < e1; k0 += cap) {
    const int k1 = (int)(k0 + cap < e1 ? k0 + cap : e1), lo = beg > k0 ? beg : (int)k0, hi = end < k1 ? end : k1;
    const bool mine = !lng && lo < hi;
    if (!__syncthreads_or(mine)) continue;  // (the readers of the last piece are done)
    const int cnt = k1 - (int)k0;
    for (int e = tid; e < cnt; e += 4 * SPR) {  // 8 loads in flight
      double v[4];
      int c[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (e + u * SPR < cnt) {
          v[u] = __ldg(A.val + k0 + e + u * SPR);
          c[u] = __ldg(A.col + k0 + e + u * SPR);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (e + u * SPR < cnt) {
          sval[e + u * SPR] = v[u];
          scol[e + u * SPR] = c[u];
        }
    }
    __syncthreads();
    spmv_walk<SCALE, SCALE ? 2 : 4>(A, scol + (lo - (int)k0), sval + (lo - (int)k0), mine ? hi - lo : 0, s0, s1, bad);
  }
  s0 += spmv_long_rows<SCALE>(A, r0, beg, len);
  spmv_store(A, r, s0 + s1, bad);
}

template <bool SCALE>
__global__ void __launch_bounds__(SPR, SCALE ? 6 : 8) spmv_block_kernel(const __grid_constant__ SpmvArgs A) {
  extern __shared__ __align__(16) unsigned char sm_sp[];
  __shared__ __align__(8) uint64_t bar;
  double* sval = reinterpret_cast<double*>(sm_sp);                   // cap + 2 values
  int32_t* scol = reinterpret_cast<int32_t*>(sval + A.cap + 2);       // cap + 4 indices
  const int tid = threadIdx.x;
  const int64_t r0 = blockIdx.x * (int64_t)SPR, r = r0 + tid;
  const int e0 = __ldg(A.rowptr + r0), e1 = __ldg(A.rowptr + (r0 + SPR < A.n ? r0 + SPR : A.n));
  if (e0 < 0 || e1 < e0 || (int64_t)e1 > A.nnz || e1 - e0 > A.cap) {
    spmv_pieces<SCALE>(A, sval, scol);
    return;
  }
  // 16-byte aligned starts at or before e0, whole 16-byte pieces before e1
  const int v0 = A.bulk ? e0 & ~1 : e0, c0 = A.bulk ? e0 & ~3 : e0;
  {
    const uint32_t bv = A.bulk ? (uint32_t)(e1 - v0) * 8u & ~15u : 0u, bc = A.bulk ? (uint32_t)(e1 - c0) * 4u & ~15u : 0u;
    if (tid == 0 && A.bulk) {
      mbar_init(&bar, 1);
      fence_mbar_init();
      mbar_arrive_expect_tx(&bar, bv + bc);
      if (bv) bulk_copy_g2s(sval, A.val + v0, bv, &bar);
      if (bc) bulk_copy_g2s(scol, A.col + c0, bc, &bar);
    }
    // what is left after the whole pieces
    for (int e = (int)(bv / 8) + tid; e < e1 - v0; e += SPR) sval[e] = __ldg(A.val + v0 + e);
    for (int e = (int)(bc / 4) + tid; e < e1 - c0; e += SPR) scol[e] = __ldg(A.col + c0 + e);
  }
  int beg, end;
  spmv_row(A, r, e0, e1, true, beg, end);
  __syncthreads();
  if (A.bulk && !mbar_wait_bounded(&bar, 0u)) {
    if (A.status) set_error(A.status, RBO_ERR_TIMEOUT, 13);
    return;
  }
  double s0 = 0.0, s1 = 0.0;
  bool bad = false;
  spmv_walk<SCALE, SCALE ? 4 : 8>(A, scol + (beg - c0), sval + (beg - v0), end - beg, s0, s1, bad);
  spmv_store(A, r, s0 + s1, bad);
}

static int spmv_dispatch_inner(const CsrDev& A, const double* dscale, const double* x,
                               const double* b, double* y, DevStatus* status, cudaStream_t st,
                               const SpmvShift& sh);

template <int LPR>
static void spmv_go(const CsrDev& A, const double* dscale, const double* x, const double* b,
                    double* y, DevStatus* status, cudaStream_t st, const SpmvShift& sh) {
  const int64_t threads = A.n * LPR;
  const int64_t blocks = (threads + 255) / 256;
  spmv_kernel<LPR><<<(unsigned)blocks, 256, 0, st>>>(A.n, A.nnz, A.rowptr, A.col, A.val, dscale, x,
                                                     b, y, status, sh);
}

static int spmv_dispatch(const CsrDev& A, const double* dscale, const double* x, const double* b,
                         double* y, DevStatus* status, cudaStream_t st, const SpmvShift& sh) {
  if (A.n <= 0) return RBO_OK;
  SpmvShift k = sh;
  if (!k.u || b) k = SpmvShift();  // (a residual has no shift)
  if (k.b == 0.0) k.uprev = nullptr;
  ProfToken tok = prof_start(st);
  int e = spmv_dispatch_inner(A, dscale, x, b, y, status, st, k);
  // algorithmic bytes: values + column indices + row pointers, x and y once each
  // (plus b, the scaling vector and the shift's vectors when used); 2 flops per
  // stored entry (+2 per row and shift term)
  const double nn = (double)A.n, nz = (double)A.nnz;
  const int terms = (k.u ? 1 : 0) + (k.uprev ? 1 : 0);
  prof_stop(tok, st, 1, 12.0 * nz + 4.0 * (nn + 1) + 16.0 * nn + (b ? 8.0 * nn : 0.0) +
                            (dscale ? 8.0 * nn : 0.0) + 8.0 * terms * nn,
            2.0 * nz + 2.0 * terms * nn);
  return e;
}

static int spmv_dispatch_inner(const CsrDev& A, const double* dscale, const double* x,
                               const double* b, double* y, DevStatus* status, cudaStream_t st,
                               const SpmvShift& sh) {
  const double avg = A.n > 0 ? (double)A.nnz / (double)A.n : 0.0;
  if (avg <= 12.0) {
    const int64_t blocks = (A.n + SPR - 1) / SPR;
    if (blocks > 0x7FFFFFFFLL) return RBO_ERR_ARG;
    // staging for a quarter more entries than the average block has (at most 3904: 46 KB)
    const int bulk = ((uintptr_t)A.col & 15) == 0 && ((uintptr_t)A.val & 15) == 0 ? 1 : 0;
    const int cap = ((int)(avg * SPR * 1.25) + 67) & ~3;
    const size_t smem = (size_t)(cap + 2) * 8 + (size_t)(cap + 4) * 4;
    SpmvArgs P{A.n, A.nnz, A.rowptr, A.col, A.val, dscale, x, b, y, status, sh,
               (uint32_t)std::min<int64_t>(A.n, (int64_t)1 << 31), cap, bulk};
    if (dscale)
      spmv_block_kernel<true><<<(unsigned)blocks, SPR, smem, st>>>(P);
    else
      spmv_block_kernel<false><<<(unsigned)blocks, SPR, smem, st>>>(P);
  } else if (avg <= 24.0)
    spmv_go<8>(A, dscale, x, b, y, status, st, sh);
  else
    spmv_go<32>(A, dscale, x, b, y, status, st, sh);
  return cudaGetLastError() == cudaSuccess ? RBO_OK : RBO_ERR_CUDA;
}

int spmv_launch(const CsrDev& A, const double* dscale, const double* x, double* y, DevStatus* status,
                cudaStream_t st, const SpmvShift& sh) {
  return spmv_dispatch(A, dscale, x, nullptr, y, status, st, sh);
}

int residual_launch(const CsrDev& A, const double* b, const double* x, double* r, DevStatus* status,
                    cudaStream_t st) {
  return spmv_dispatch(A, nullptr, x, b, r, status, st, SpmvShift());
}

__global__ void scale_columns_kernel(int64_t n, int64_t nnz, const int32_t* __restrict__ col,
                                     const double* __restrict__ val, const double* __restrict__ ds,
                                     double* __restrict__ out) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (; j < nnz; j += stride) {
    const int32_t c = col[j];
    out[j] = (c >= 0 && (int64_t)c < n) ? val[j] * ds[c] : 0.0;
  }
}

int scale_columns_launch(const CsrDev& A, const double* dscale, double* val_out, cudaStream_t st) {
  if (A.nnz <= 0) return RBO_OK;
  int64_t blocks = std::min<int64_t>((A.nnz + 255) / 256, 65535LL * 16);
  scale_columns_kernel<<<(unsigned)blocks, 256, 0, st>>>(A.n, A.nnz, A.col, A.val, dscale, val_out);
  return cudaGetLastError() == cudaSuccess ? RBO_OK : RBO_ERR_CUDA;
}

__global__ void jacobi_kernel(int64_t n, int64_t nnz, const int32_t* __restrict__ rowptr,
                              const int32_t* __restrict__ col, const double* __restrict__ val,
                              double* __restrict__ ds, DevStatus* status) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double dia = 0.0;
  int beg = rowptr[i], end = rowptr[i + 1];
  if (beg < 0 || end < beg || (int64_t)end > nnz) end = beg;
  for (int j = beg; j < end; ++j)
    if (col[j] == (int32_t)i) dia = val[j];
  if (dia == 0.0) {
    set_error(status, RBO_ERR_ARG, 10);
    ds[i] = 0.0;
  } else {
    ds[i] = 1.0 / dia;
  }
}

int jacobi_launch(const CsrDev& A, double* dscale, DevStatus* status, cudaStream_t st) {
  if (A.n <= 0) return RBO_OK;
  jacobi_kernel<<<(unsigned)((A.n + 255) / 256), 256, 0, st>>>(A.n, A.nnz, A.rowptr, A.col, A.val, dscale,
                                                                status);
  return cudaGetLastError() == cudaSuccess ? RBO_OK : RBO_ERR_CUDA;
}

// y = Q z (accumulate = 0) or y += Q z: one thread per row, z in shared memory
__global__ void gemv_update_kernel(int64_t n, int k, const double* __restrict__ Q, int64_t ldq,
                                   const double* __restrict__ z, double* __restrict__ y,
                                   int accumulate) {
  __shared__ double zs[256];
  for (int t = threadIdx.x; t < k; t += blockDim.x) zs[t] = z[t];
  __syncthreads();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0;
  for (int c = 0; c < k; ++c) s = fma(Q[i + c * ldq], zs[c], s);
  y[i] = accumulate ? y[i] + s : s;
}

// x += D t  (D = diag(ds), or the identity when ds is null)
__global__ void axpy_scaled_kernel(int64_t n, const double* __restrict__ ds,
                                   const double* __restrict__ t, double* __restrict__ x) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  x[i] += ds ? ds[i] * t[i] : t[i];
}

int axpy_scaled_launch(int64_t n, const double* ds, const double* t, double* x, cudaStream_t st) {
  if (n <= 0) return RBO_OK;
  axpy_scaled_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, ds, t, x);
  return cudaGetLastError() == cudaSuccess ? RBO_OK : RBO_ERR_CUDA;
}

// Newton-basis step: out += a u + b uprev (uprev may be null when b = 0)
int gemv_update_launch(int64_t n, int k, const double* Q, int64_t ldq, const double* z, double* y,
                       int accumulate, cudaStream_t st) {
  if (n <= 0 || k <= 0) return RBO_OK;
  if (k > 256) return RBO_ERR_ARG;
  gemv_update_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, k, Q, ldq, z, y, accumulate);
  return cudaGetLastError() == cudaSuccess ? RBO_OK : RBO_ERR_CUDA;
}

__global__ void scale_vec_kernel(int64_t n, const double* __restrict__ ds, const double* __restrict__ y,
                                 double* __restrict__ x, int mode) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double v = y[i];
  if (ds) v = mode == 0 ? v * ds[i] : v / ds[i];
  x[i] = v;
}

int scale_vec_launch(int64_t n, const double* dscale, const double* y, double* x, int mode,
                     cudaStream_t st) {
  if (n <= 0) return RBO_OK;
  scale_vec_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, dscale, y, x, mode);
  return cudaGetLastError() == cudaSuccess ? RBO_OK : RBO_ERR_CUDA;
}

}  // namespace rbo

namespace rbo {

// ---- SELL-32: the short-row matrices of the MPK in sliced ELL form -------------------
// A warp owns a slice of 32 rows and a lane its row: slot j of the slice is one
// coalesced 256-byte value load and 128-byte index load for the whole warp, and the
// slots of a row are summed in two interleaved chains (even, odd j) added at the end, a
// fixed order.  Padding slots (value 0, the row's own index) cost a multiply-add.

__global__ void sell_width_kernel(int64_t n, int64_t nnz, const int32_t* __restrict__ rowptr,
                                  int32_t* __restrict__ width, DevStatus* status) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t k = t >> 5;
  const int lane = (int)(t & 31);
  const int64_t nsl = (n + 31) / 32;
  if (k >= nsl) return;  // whole warps (nsl * 32 threads are launched)
  const int64_t r = k * 32 + lane;
  int len = 0;
  if (r < n) {
    const int beg = rowptr[r], end = rowptr[r + 1];
    if (beg < 0 || end < beg || (int64_t)end > nnz) {
      if (status) set_error(status, RBO_ERR_ARG, 11);
    } else {
      len = end - beg;
    }
  }
  len = __reduce_max_sync(0xffffffffu, len);
  if (lane == 0) width[k] = len;
}

__global__ void sell_fill_kernel(int64_t n, int64_t nnz, const int32_t* __restrict__ rowptr,
                                 const int32_t* __restrict__ ccol, const double* __restrict__ cval,
                                 const int64_t* __restrict__ soff, int32_t* __restrict__ col,
                                 double* __restrict__ val, DevStatus* status) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t k = t >> 5;
  const int lane = (int)(t & 31);
  if (k >= (n + 31) / 32) return;
  const int64_t r = k * 32 + lane;
  const int64_t off = soff[k];
  const int w = (int)((soff[k + 1] - off) / 32);
  int beg = 0, len = 0;
  if (r < n) {
    beg = rowptr[r];
    const int end = rowptr[r + 1];
    if (beg >= 0 && end >= beg && (int64_t)end <= nnz) len = end - beg;
  }
  const int32_t self = (int32_t)(r < n ? r : 0);
  for (int j = 0; j < w; ++j) {
    int32_t c = self;
    double v = 0.0;
    if (j < len) {
      const int32_t cj = ccol[beg + j];
      if (cj < 0 || (int64_t)cj >= n) {
        if (status) set_error(status, RBO_ERR_ARG, 12);
      } else {
        c = cj;
        v = cval[beg + j];
      }
    }
    col[off + (int64_t)j * 32 + lane] = c;
    val[off + (int64_t)j * 32 + lane] = v;
  }
}

__global__ void __launch_bounds__(256, 6) spmv_sell_kernel(int64_t n, int64_t nsl, const int64_t* __restrict__ soff,
                                                           const int32_t* __restrict__ col,
                                                           const double* __restrict__ val,
                                                           const double* __restrict__ x, double* __restrict__ y,
                                                           SpmvShift sh) {
  // one slice per warp (the grid covers the matrix): every warp's loads are in flight
  // at once; slices of up to 8 slots load all indices and values before the gathers
  const int lane = threadIdx.x & 31;
  const int64_t k = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  if (k >= nsl) return;
  const int64_t off = __ldg(soff + k);
  const int w = (int)((__ldg(soff + k + 1) - off) >> 5);
  const int32_t* cp = col + off + lane;
  const double* vp = val + off + lane;
  double s0 = 0.0, s1 = 0.0;
  if (w <= 8) {
    int32_t c[8];
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      c[j] = j < w ? __ldg(cp + 32 * j) : 0;
      v[j] = j < w ? __ldg(vp + 32 * j) : 0.0;
    }
    double xv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) xv[j] = j < w ? __ldg(x + c[j]) : 0.0;
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      if (j < w) s0 = fma(v[j], xv[j], s0);
      if (j + 1 < w) s1 = fma(v[j + 1], xv[j + 1], s1);
    }
  } else {
    for (int j = 0; j < w; ++j) {
      const double vv = __ldg(vp + 32 * j), xx = __ldg(x + __ldg(cp + 32 * j));
      if (j & 1) s1 = fma(vv, xx, s1);
      else s0 = fma(vv, xx, s0);
    }
  }
  const int64_t r = k * 32 + lane;
  if (r < n) y[r] = shifted(s0 + s1, sh, r);
}

}  // namespace rbo

namespace rbo {

int sell_build(const CsrDev& A, int64_t cap_slots, int64_t* soff, int32_t* width, int32_t* col,
               double* val, DevStatus* status, cudaStream_t st, SellDev* out) {
  *out = SellDev();
  if (A.n <= 0) return RBO_OK;
  const int64_t nsl = (A.n + 31) / 32;
  const int64_t threads = nsl * 32;
  sell_width_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(A.n, A.nnz, A.rowptr, width, status);
  if (cudaGetLastError() != cudaSuccess) return RBO_ERR_CUDA;
  std::vector<int32_t> wh((size_t)nsl);
  std::vector<int64_t> oh((size_t)nsl + 1);
  if (cudaMemcpyAsync(wh.data(), width, (size_t)nsl * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return RBO_ERR_CUDA;
  oh[0] = 0;
  for (int64_t k = 0; k < nsl; ++k) oh[(size_t)k + 1] = oh[(size_t)k] + 32 * (int64_t)wh[(size_t)k];
  if (oh[(size_t)nsl] > cap_slots) return RBO_OK;  // too much padding: stay with CSR
  if (cudaMemcpyAsync(soff, oh.data(), (size_t)(nsl + 1) * 8, cudaMemcpyHostToDevice, st) != cudaSuccess)
    return RBO_ERR_CUDA;
  sell_fill_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(A.n, A.nnz, A.rowptr, A.col, A.val, soff,
                                                                      col, val, status);
  if (cudaGetLastError() != cudaSuccess) return RBO_ERR_CUDA;
  // the host copy of the offsets must outlive the asynchronous upload
  if (cudaStreamSynchronize(st) != cudaSuccess) return RBO_ERR_CUDA;
  out->n = A.n;
  out->nslices = nsl;
  out->soff = soff;
  out->col = col;
  out->val = val;
  return RBO_OK;
}

int spmv_sell_launch(const SellDev& S, int64_t nnz, const double* x, double* y, cudaStream_t st,
                     const SpmvShift& sh) {
  if (S.n <= 0) return RBO_OK;
  SpmvShift k = sh;
  if (!k.u) k = SpmvShift();
  if (k.b == 0.0) k.uprev = nullptr;
  const int64_t blocks = (S.nslices + 7) / 8;
  if (blocks > 0x7FFFFFFFLL) return RBO_ERR_ARG;
  ProfToken tok = prof_start(st);
  spmv_sell_kernel<<<(unsigned)blocks, 256, 0, st>>>(S.n, S.nslices, S.soff, S.col, S.val, x, y, k);
  // algorithmic bytes and flops as for the CSR kernel (the stored entries, not the padding)
  const double nn = (double)S.n, nz = (double)nnz;
  const int terms = (k.u ? 1 : 0) + (k.uprev ? 1 : 0);
  prof_stop(tok, st, 1, 12.0 * nz + 4.0 * (nn + 1) + 16.0 * nn + 8.0 * terms * nn, 2.0 * nz + 2.0 * terms * nn);
  return cudaGetLastError() == cudaSuccess ? RBO_OK : RBO_ERR_CUDA;
}

}  // namespace rbo
