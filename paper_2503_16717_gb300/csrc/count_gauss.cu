// The dense half of a Count-Gauss sketch: G times the Count stage of a row pass (the sum of its
// group partials, di x k), and the small factorisations of the product for shapes that the
// cluster kernel (skb2.cu) does not take.
//
// Every entry of G is generated (SplitMix64 and a float32 Box-Muller) where it is used, about 60
// instructions each: one warp per row of G, lanes over the inner rows, 8 columns per entry
// generated, all SMs (d = 128, di = 1000, k = 5: sketch of 400001 rows 266 us a call; 1405 us with the
// product in the last CTA of the pass, 128 threads, an entry per column).  Sums run over a lane's
// inner rows and then over the lanes, a fixed order.
#include <algorithm>
#include <mutex>

#include "rowpass_common.cuh"

namespace rbo {

constexpr int CG_NT = 256;

// S[t] = sum of the partials in order, t < L
__global__ void cg_sum_kernel(const double* __restrict__ part, int nparts, int L, double* __restrict__ S,
                              const DevStatus* status) {
  const int t = blockIdx.x * CG_NT + threadIdx.x;
  if (t >= L || read_code(status) != 0) return;
  double s = 0.0;
  for (int g0 = 0; g0 < nparts; g0 += 16) {  // 16 loads in flight
    double v[16];
#pragma unroll
    for (int g = 0; g < 16; ++g) v[g] = g0 + g < nparts ? part[(size_t)(g0 + g) * L + t] : 0.0;
#pragma unroll
    for (int g = 0; g < 16; ++g) s += v[g];
  }
  S[t] = s;
}

// out (d x k) = G S (di x k), a row of G per warp
__global__ void cg_product_kernel(const double* __restrict__ S, int di, int d, int k, uint64_t seed,
                                  double* __restrict__ out, const DevStatus* status) {
  const int row = blockIdx.x * (CG_NT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= d || read_code(status) != 0) return;
  for (int c0 = 0; c0 < k; c0 += 8) {
    double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int j = lane; j < di; j += 32) {
      const double g = (double)gauss_entry(seed, (uint64_t)j, row, d);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (c0 + u < k) s[u] = fma(g, S[j + (size_t)(c0 + u) * di], s[u]);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (c0 + u < k) {
        const double v = warp_sum(s[u]);
        if (lane == 0) out[row + (size_t)(c0 + u) * d] = v;
      }
  }
}

int count_gauss_launch(const double* part, int nparts, int di, int d, int k, uint64_t seed, double* S, double* out,
                       DevStatus* status, cudaStream_t st, int* launches) {
  const int L = di * k;
  cg_sum_kernel<<<(L + CG_NT - 1) / CG_NT, CG_NT, 0, st>>>(part, nparts, L, S, status);
  cg_product_kernel<<<(d + CG_NT / 32 - 1) / (CG_NT / 32), CG_NT, 0, st>>>(S, di, d, k, seed, out, status);
  if (launches) *launches += 2;
  return note_cuda(cudaGetLastError());
}

// The epilogue of a pass on its finished sketch v (d x b)
__global__ void __launch_bounds__(CG_NT) sketch_epilogue_kernel(const __grid_constant__ PassDev P,
                                                                const double* __restrict__ v) {
  extern __shared__ __align__(16) double red[];
  __shared__ int s_flag;
  if (read_code(P.status) != 0) return;
  for (int t = threadIdx.x; t < P.L; t += CG_NT) red[t] = v[t];
  __syncthreads();
  run_epilogue(P, red, red + ((P.L + 1) & ~1), &s_flag);
}

int sketch_epilogue_launch(const Epilogue& epi, const double* v, int d, int k, DevStatus* status, cudaStream_t st,
                           int* launches) {
  PassDev P = PassDev();
  P.p.b = k;
  P.p.sk_d = d;
  P.p.epi = epi;
  P.L = d * k;
  P.status = status;
  const size_t smem = ((size_t)P.L + 2 + epilogue_doubles(P.p)) * 8;
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if ((long long)smem + 64 > optin) return RBO_ERR_ARG;
  const int e = note_cuda(
      cudaFuncSetAttribute(sketch_epilogue_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 64));
  if (e != RBO_OK) return e;
  sketch_epilogue_kernel<<<1, CG_NT, smem, st>>>(P, v);
  if (launches) ++*launches;
  return note_cuda(cudaGetLastError());
}

}  // namespace rbo
