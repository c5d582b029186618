// The small dense work on a panel's sketch, on a cluster of 8 CTAs: the Householder factor
// R of RandHH (one-stage, Section 5.2), or the sketched BCGS2 with Householder intra step of
// the two-stage preprocessing (Section 7.2): v (d x k) against the sketched basis qs
// (d x poff) of the big panel, giving T(:, panel) and the panel's sketched basis columns.
// v is the sum of the sketch pass's group partials (fixed order).
//
// The work is small but float64, and one SM does 2 float64 FMAs per cycle: the four
// products with qs take 4 d poff k of them, 160 us of one SM at d = 404, poff = 40,
// k = 10.  Here every CTA owns d / 8 rows of v and qs in its shared memory.  What crosses
// the rows (the products qs^T v, the dot products of a Householder step, V^T V) is summed
// from the CTAs' partials over distributed shared memory in a fixed order, one cluster
// barrier each; everything else is local.  The Householder step of column j needs one
// exchange: the dot products of the column below row j with all later columns, and row j,
// determine the reflector and its application.  Q comes from the compact WY form
// I - V T V^T (Schreiber and Van Loan 1989).  Measured 13 us (d = 244, k = 5, the Householder
// factor) to 19 us (with a sketched basis) between launches of one call, 25 and 39 us a launch
// serialised with cold caches; a chain of cluster barriers and float64 latencies.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "device_common.cuh"
#include "small_dense.cuh"

namespace rbo {
namespace cg = cooperative_groups;

constexpr int SKB2_CTAS = 8;  // (the exchange sums eight partials)
constexpr int SKB2_NT = 256;

struct Skb2Dev {
  const double* v;   // nparts partials of d x k, `stride` apart
  int nparts;
  int64_t stride;
  double* qs;        // d x K sketched basis, columns poff.. written; null: R only
  double* T;         // K x K
  int d, k, K, poff, m;  // m: rows per CTA
  int stage, block;
  DevStatus* status;
};

__global__ void __cluster_dims__(SKB2_CTAS, 1, 1) __launch_bounds__(SKB2_NT) skb2_kernel(const Skb2Dev P) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double s_col[4];  // beta, v0, alpha sign, R_jj of the current column
  cg::cluster_group cl = cg::this_cluster();
  // every CTA of the cluster reads the same code: it only changes between launches here
  if (read_code(P.status) != 0) return;
  const int tid = threadIdx.x, rank = (int)cl.block_rank();
  const int k = P.k, pp = P.poff, d = P.d, K = P.K, m = P.m;
  const int r0 = rank * m, nr = max(0, min(m, d - r0));
  const int np = max(max(pp, k), 2) * k;   // length of one partial
  double* a = sm;                          // m x k: v, then the reflectors
  double* q = a + m * k;                   // m x pp
  double* part = q + m * pp;               // 2 x np: this CTA's partials (two buffers)
  double* c1 = part + 2 * np;              // np
  double* cs = c1 + np;                    // np: sum of both projections
  double* R = cs + np;                     // k x k
  double* Vt = R + k * k;                  // k x k: rows 0..k-1 of V
  double* G = Vt + k * k;                  // k x k: V^T V, then T
  double* W = G + k * k;                   // k x k
  double* beta = W + k * k;                // k

  for (int e = tid; e < nr * k; e += SKB2_NT) {
    const double* v = P.v + r0 + e % nr + (size_t)(e / nr) * d;
    double s = 0.0;
    for (int g0 = 0; g0 < P.nparts; g0 += 16) {  // 16 loads in flight, summed in order
      double t[16];
#pragma unroll
      for (int g = 0; g < 16; ++g) t[g] = g0 + g < P.nparts ? __ldcg(v + (int64_t)(g0 + g) * P.stride) : 0.0;
#pragma unroll
      for (int g = 0; g < 16; ++g)
        if (g0 + g < P.nparts) s += t[g];
    }
    a[(e % nr) + (e / nr) * m] = s;
  }
  for (int e = tid; e < nr * pp; e += SKB2_NT) q[(e % nr) + (e / nr) * m] = P.qs[r0 + e % nr + (size_t)(e / nr) * d];
  for (int e = tid; e < k * k; e += SKB2_NT) R[e] = 0.0;
  for (int e = tid; e < np; e += SKB2_NT) cs[e] = 0.0;
  __syncthreads();

  int buf = 0;
  // out[e] = sum over the CTAs of their part[buf][e], e < cnt (fixed order); all threads
  auto exchange = [&](double* out, int cnt) {
    cl.sync();
    for (int e = tid; e < cnt; e += SKB2_NT) {
      double v[SKB2_CTAS];
#pragma unroll
      for (int r = 0; r < SKB2_CTAS; ++r) v[r] = cl.map_shared_rank(part, r)[buf * np + e];
      out[e] = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    buf ^= 1;
    __syncthreads();
  };

  for (int pass = 0; pass < 2 && pp > 0; ++pass) {  // c = qs^T v; v -= qs c, twice
    for (int e = tid; e < pp * k; e += SKB2_NT) {
      const double* qc = q + (e % pp) * m;
      const double* ac = a + (e / pp) * m;
      double s0 = 0.0, s1 = 0.0;
      int r = 0;
      for (; r + 1 < nr; r += 2) {
        s0 = fma(qc[r], ac[r], s0);
        s1 = fma(qc[r + 1], ac[r + 1], s1);
      }
      if (r < nr) s0 = fma(qc[r], ac[r], s0);
      part[buf * np + e] = s0 + s1;
    }
    exchange(c1, pp * k);
    for (int e = tid; e < pp * k; e += SKB2_NT) cs[e] += c1[e];
    for (int e = tid; e < nr * k; e += SKB2_NT) {
      const int r = e % nr, c = e / nr;
      double s0 = a[r + c * m], s1 = 0.0;
      int i = 0;
      for (; i + 1 < pp; i += 2) {
        s0 = fma(-q[r + i * m], c1[i + c * pp], s0);
        s1 = fma(-q[r + (i + 1) * m], c1[i + 1 + c * pp], s1);
      }
      if (i < pp) s0 = fma(-q[r + i * m], c1[i + c * pp], s0);
      a[r + c * m] = s0 + s1;
    }
    __syncthreads();
  }

  // Householder: column j over the rows below j (global row index r0 + r)
  const int lane = tid & 31, warp = tid >> 5;
  for (int j = 0; j < k; ++j) {
    const int lo = min(max(j + 1 - r0, 0), nr);  // first local row below row j
    double* mine = part + buf * np;
    for (int c = j + warp; c < k; c += SKB2_NT / 32) {
      double s = 0.0;
      for (int r = lo + lane; r < nr; r += 32) s = fma(a[r + j * m], a[r + c * m], s);
      s = warp_sum(s);
      if (lane == 0) mine[c] = s;
    }
    for (int c = tid; c < k; c += SKB2_NT) {  // row j from its owner
      mine[k + c] = (j >= r0 && j < r0 + nr) ? a[(j - r0) + c * m] : 0.0;
      if (c < j) mine[c] = 0.0;
    }
    exchange(c1, 2 * k);
    if (tid == 0) {
      const double rest = c1[j], x0 = c1[k + j];
      const double sq = rest + x0 * x0, s = x0 >= 0.0 ? 1.0 : -1.0;
      // 2 / v^T v = 1 / (alpha (alpha + |x0|)); the fast forms inside the range where that
      // product is normal
      double alpha, v0, b2;
      if (sq > 1e-280 && sq < 1e280) {
        double inva;
        sqrt_and_inverse(sq, alpha, inva);
        v0 = x0 + s * alpha;
        b2 = fast_reciprocal(alpha * fabs(v0));
      } else {
        alpha = sqrt(sq);
        v0 = x0 + s * alpha;
        b2 = alpha == 0.0 ? 0.0 : 1.0 / alpha / fabs(v0);
      }
      s_col[0] = beta[j] = b2;
      s_col[1] = v0;
      R[j + j * k] = -s * alpha;
    }
    __syncthreads();
    const double bj = s_col[0], v0 = s_col[1];
    for (int c = tid; c < k; c += SKB2_NT) {
      Vt[j + c * k] = c < j ? c1[k + c] : (c == j ? v0 : 0.0);
      if (c > j) R[j + c * k] = c1[k + c] - (c1[c] + v0 * c1[k + c]) * bj * v0;
    }
    for (int e = tid; e < (nr - lo) * (k - 1 - j); e += SKB2_NT) {
      const int r = lo + e % (nr - lo), c = j + 1 + e / (nr - lo);
      const double w = (c1[c] + v0 * c1[k + c]) * bj;
      a[r + c * m] = fma(-w, a[r + j * m], a[r + c * m]);
    }
    if (j >= r0 && j < r0 + nr)
      for (int c = j + tid; c < k; c += SKB2_NT)
        a[(j - r0) + c * m] = c == j ? v0 : c1[k + c] - (c1[c] + v0 * c1[k + c]) * bj * v0;
    __syncthreads();
  }
  if (P.qs != nullptr) {
    // V^T V (strict upper triangle), V(i, j) = 0 above row j
    for (int t = warp; t < k * k; t += SKB2_NT / 32) {
      const int i = t % k, c = t / k;
      double s = 0.0;
      if (i < c)
        for (int r = min(max(c - r0, 0), nr) + lane; r < nr; r += 32) s = fma(a[r + i * m], a[r + c * m], s);
      s = warp_sum(s);
      if (lane == 0) part[buf * np + t] = s;
    }
    exchange(G, k * k);
    // T of the WY form in place of G: T_jj = beta_j, T(:j, j) = -beta_j T(:j, :j) (V^T v_j)(:j)
    for (int j = 0; j < k; ++j) {
      double t = 0.0;
      if (tid < j)
        for (int l = tid; l < j; ++l) t = fma(G[tid + l * k], G[l + j * k], t);
      __syncthreads();
      if (tid < j) G[tid + j * k] = -beta[j] * t;
      if (tid == j) G[j + j * k] = beta[j];
      __syncthreads();
    }
    // W = T Vt^T (Vt lower triangular)
    for (int e = tid; e < k * k; e += SKB2_NT) {
      const int i = e % k, c = e / k;
      double s = 0.0;
      for (int l = i; l <= c; ++l) s = fma(G[i + l * k], Vt[c + l * k], s);
      W[e] = s;
    }
    __syncthreads();
    // Q = I - V W with the signs that make diag(R) >= 0
    for (int e = tid; e < nr * k; e += SKB2_NT) {
      const int r = e % nr, c = e / nr, gr = r0 + r;
      double s = gr == c ? 1.0 : 0.0;
      for (int l = 0; l < k && l <= gr; ++l) s = fma(-a[r + l * m], W[l + c * k], s);
      P.qs[gr + (size_t)(pp + c) * d] = R[c + c * k] < 0.0 ? -s : s;
    }
  }
  if (rank == 0) {
    for (int e = tid; e < pp * k; e += SKB2_NT) P.T[e % pp + (size_t)(pp + e / pp) * K] = cs[e];
    for (int e = tid; e < k * k; e += SKB2_NT) {
      const int i = e % k, c = e / k;
      P.T[(pp + i) + (size_t)(pp + c) * K] = R[i + i * k] < 0.0 ? -R[e] : R[e];
    }
    if (tid == 0) {
      const int bad = tri_rank_deficient(R, k);
      if (bad >= 0) set_breakdown(P.status, P.block, pp + bad, P.stage);
    }
  }
  cl.sync();  // no CTA leaves while another may still read its partials
}

static std::mutex g_skb2_mu;
static int g_skb2_set[64] = {};

// Whether the cluster kernel serves this shape (otherwise the epilogue of the pass does)
bool skb2_supported(int d, int k, int poff) { return k <= 16 && d >= k && poff <= 64 && d <= 1024; }

int skb2_launch(const double* v, int nparts, int64_t stride, double* qs, double* T, int d, int k, int K, int poff,
                int stage, int block, DevStatus* status, cudaStream_t st, int* launches) {
  if (!skb2_supported(d, k, poff)) return RBO_ERR_ARG;
  Skb2Dev P{v, nparts, stride, qs, T, d, k, K, poff, (d + SKB2_CTAS - 1) / SKB2_CTAS, stage, block, status};
  const int np = std::max(std::max(poff, k), 2) * k;
  const size_t smem = ((size_t)P.m * (k + poff) + 4 * (size_t)np + 4 * (size_t)k * k + k) * 8;
  int dev = 0;
  cudaGetDevice(&dev);
  {
    std::lock_guard<std::mutex> lk(g_skb2_mu);
    if (dev >= 0 && dev < 64 && !g_skb2_set[dev]) {
      const int e = note_cuda(cudaFuncSetAttribute(skb2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
      if (e != RBO_OK) return e;
      g_skb2_set[dev] = 1;
    }
  }
  skb2_kernel<<<SKB2_CTAS, SKB2_NT, smem, st>>>(P);
  if (launches) ++*launches;
  return note_cuda(cudaGetLastError());
}

}  // namespace rbo
