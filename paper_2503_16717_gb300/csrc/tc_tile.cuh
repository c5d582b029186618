// Warp-level tile products of the row passes on the tensor cores (tc_fixed.cuh): a Gram
// item (16 columns of Z against 8 columns of Y' over a chunk of tile rows) and the update
// y - x C of 16 tile rows.
//
// Tiles: blocks of 16 rows, a column of a block is one 128-byte line, its 16-byte chunks
// (two rows) permuted by the column: chunk j of column c sits at j ^ (c % 8).  This is
// what a tensor copy of a (16 rows x columns) box with the 128-byte swizzle writes, and
// both access patterns below are free of bank conflicts in it.  Columns are padded with
// zeros to a multiple of 8 (blocks of a multiple of 1024 bytes), the left operand of a
// product with digits of C to a multiple of 16.
#pragma once

#include "tc_fixed.cuh"

namespace rbo {

// The first K step of a sum is apart: its products take the starting value as their addend,
// which saves setting 28 accumulators per sum (2^22 x 61, one-stage: P1 504 -> 484 us, update +
// Gram 593 -> 570 us, all 40.1 -> 37.9 ms).
struct FxTrue { static constexpr bool value = true; };    // first step of a sum
struct FxFalse { static constexpr bool value = false; };

struct TcTile {
  const unsigned char* base;  // 1024-byte aligned
  int blk;                    // bytes of a 16-row block
  // byte offset of (row r, column c)
  __device__ __forceinline__ static int off(int blk, int r, int c) {
    return (r >> 4) * blk + c * 128 + ((((r >> 1) & 7) ^ (c & 7)) << 4) + ((r & 1) << 3);
  }
};
__host__ __device__ inline int tc_blk_bytes(int cols, int pad) { return ((cols + pad - 1) & ~(pad - 1)) * 128; }
__device__ __forceinline__ double tc_ld(const unsigned char* p) { return *reinterpret_cast<const double*>(p); }
__device__ __forceinline__ double2 tc_ld2(const unsigned char* p) { return *reinterpret_cast<const double2*>(p); }

// Joins the level sums of an item into its float64 slots.  E0, E1: scales of Z columns g
// and g + 8; Eb: of Y column g (this lane's).
__device__ __forceinline__ void tc_gram_flush(float (&acc)[7][4], bool small, int E0, int E1, int Eb, bool both,
                                              double* acc_out) {
  const int lane = threadIdx.x & 31, t = lane & 3;
  fx_ints(acc, small);
  const int Ea = __shfl_sync(0xffffffffu, Eb, 8 * t), Ec = __shfl_sync(0xffffffffu, Eb, 8 * t + 4);
  acc_out[lane] = fma(fx_join(acc, 0), fx_weight(E0, Ea), acc_out[lane]);
  acc_out[32 + lane] = fma(fx_join(acc, 1), fx_weight(E0, Ec), acc_out[32 + lane]);
  if (both) {
    acc_out[64 + lane] = fma(fx_join(acc, 2), fx_weight(E1, Ea), acc_out[64 + lane]);
    acc_out[96 + lane] = fma(fx_join(acc, 3), fx_weight(E1, Ec), acc_out[96 + lane]);
  }
}

// Whether an item has an entry whose digits are not good enough.  In units of a product of two
// top digits, a chunk of k rows is off by at most 2^-38.6 k (the pairs left out, the truncated
// bits), whatever its terms; the sum S of |d_x d_y| over the top digits is the sum of the terms'
// sizes to within the lower digits.  Where S >= 16 k the chunk is off by at most 2^-41 of that sum,
// less than 4096 roundings of a float64 sum.  (The largest value of a column has a top digit of 64
// to 128; chunks of Gaussian columns lie ten times above the line.)  Below it the chunk is summed by
// FMAs.  The sums S cost 5 % (60 x 5 columns at 4 million rows 757 -> 790 us), so they are for Grams
// that are results themselves: in the orthogonalization, whose errors are measured against the
// norms of the columns, the plain items serve.  Whole warp.
__device__ __forceinline__ bool tc_gram_small(const float (&sizes)[4], int nks, int E0, int E1, int Eb) {
  const int t = threadIdx.x & 3;
  const int Ea = __shfl_sync(0xffffffffu, Eb, 8 * t), Ec = __shfl_sync(0xffffffffu, Eb, 8 * t + 4);
  const float lim = (float)(256 * nks);
  const bool z0 = E0 != FX_EZERO, z1 = E1 != FX_EZERO, ya = Ea != FX_EZERO, yc = Ec != FX_EZERO;
  return (sizes[0] < lim && z0 && ya) || (sizes[1] < lim && z0 && yc) || (sizes[2] < lim && z1 && ya) ||
         (sizes[3] < lim && z1 && yc);
}

// The same item by float64 FMAs, for the guarded Gram, where it may run often: the outputs dealt to
// the lanes, up to four each (an outlier in every chunk of 59 x 5 columns: 355 us at 400001 rows;
// two rows and two columns of 16 x 8 a lane, 440).  Not inlined: the digit products keep their
// registers.  Whole warp.
static __device__ __noinline__ void tc_gram_fma(const TcTile xt, const TcTile yt, int ax, int zr, int b, int mt, int nt,
                                                int ntiles, int b0, int nks, double* acc_out) {
  const int lane = threadIdx.x & 31, zw = min(16, zr - 16 * mt);
  __syncwarp();
  for (int h = 0; h < ntiles; ++h) {
    const int c0 = 8 * (nt + h), cnt = zw * min(8, b - c0);
    const unsigned char *px[4], *py[4];
    int zc[4], yc[4], xb[4];
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int o = min(lane + 32 * u, max(cnt, 1) - 1), z = 16 * mt + o % zw;
      yc[u] = min(c0 + o / zw, b - 1);
      zc[u] = z < ax ? z : z - ax;
      xb[u] = z < ax ? xt.blk : yt.blk;
      px[u] = (z < ax ? xt.base : yt.base) + b0 * xb[u];
      py[u] = yt.base + b0 * yt.blk;
    }
    for (int r = 0; r < 16 * nks; ++r)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (32 * u < cnt)
          s[u] = fma(tc_ld(px[u] + TcTile::off(xb[u], r, zc[u])), tc_ld(py[u] + TcTile::off(yt.blk, r, yc[u])), s[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int o = lane + 32 * u;
      if (o < cnt) {
        const int zi = o % zw, c = o / zw;
        acc_out[h * 128 + (2 * (zi >> 3) + (c & 1)) * 32 + 4 * (zi & 7) + (c >> 1)] += s[u];
      }
    }
  }
  __syncwarp();
}

// acc_out (NT times 4 x 32 doubles, this warp's own) += Z(:, 16 mt ..)^T Y(:, 8 nt ..) over the
// nks blocks of 16 rows from block b0, for the NT column tiles from nt; Z = [X (ax columns, tile
// xt), Y (tile yt)], zr columns (the last one stands in for columns past the end, whose sums are
// not read).
// Lane (g, t) = (lane / 4, lane % 4) owns rows 4t..4t+3 of every block for the columns g,
// g + 8 of Z and g of Y: the order of the rows inside a step is the same for both
// operands, which is all a contraction needs, and makes every load 16 bytes.
// acc_out[o * 32 + lane] belongs to Z column 16 mt + g + 8 (o / 2), Y column 8 nt + 2t + o % 2.
// GUARD: chunks whose large values do not meet are summed by FMAs (tc_gram_small).
template <int NT, bool GUARD>
static __device__ __forceinline__ void tc_gram_item(const TcTile xt, const TcTile yt, int ax, int zr, int b,
                                                    int mt, int nt, int b0, int nks, double* acc_out) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int i0 = 16 * mt;
  const int za = min(i0 + g, zr - 1), zc = min(i0 + 8 + g, zr - 1);
  const int blk0 = za < ax ? xt.blk : yt.blk, blk1 = zc < ax ? xt.blk : yt.blk;
  const int ca = za < ax ? za : za - ax, cc = zc < ax ? zc : zc - ax;
  const unsigned char* z0 = (za < ax ? xt.base : yt.base) + b0 * blk0 + ca * 128;
  const unsigned char* z1 = (zc < ax ? xt.base : yt.base) + b0 * blk1 + cc * 128;
  const int oa = ((2 * t) ^ (ca & 7)) << 4, ob = ((2 * t) ^ (cc & 7)) << 4;
  const unsigned char* y0[NT];
  int oy[NT];
#pragma unroll
  for (int h = 0; h < NT; ++h) {
    const int yc = min(8 * (nt + h) + g, b - 1);
    y0[h] = yt.base + b0 * yt.blk + yc * 128;
    oy[h] = ((2 * t) ^ (yc & 7)) << 4;
  }
  FxMax m0, m1, mb[NT];
  for (int ks = 0; ks < nks; ++ks) {
    const unsigned char *pa = z0 + ks * blk0, *pc = z1 + ks * blk1;
    const double2 u0 = tc_ld2(pa + oa), u1 = tc_ld2(pa + (oa ^ 16));
    const double2 w0 = tc_ld2(pc + ob), w1 = tc_ld2(pc + (ob ^ 16));
#pragma unroll
    for (int h = 0; h < NT; ++h) {
      const unsigned char* py = y0[h] + ks * yt.blk;
      const double2 v0 = tc_ld2(py + oy[h]), v1 = tc_ld2(py + (oy[h] ^ 16));
      mb[h].add(v0.x, v0.y);
      mb[h].add(v1.x, v1.y);
    }
    m0.add(u0.x, u0.y);
    m0.add(u1.x, u1.y);
    m1.add(w0.x, w0.y);
    m1.add(w1.x, w1.y);
  }
  m0.reduce4();
  m1.reduce4();
  const int E0 = m0.scale(), E1 = m1.scale();
  int Eb[NT];
  bool out = E0 == 0 || E1 == 0;
#pragma unroll
  for (int h = 0; h < NT; ++h) {
    mb[h].reduce4();
    Eb[h] = mb[h].scale();
    out = out || Eb[h] == 0;
  }
  if (__any_sync(0xffffffffu, out)) {
    if constexpr (GUARD) {
      tc_gram_fma(xt, yt, ax, zr, b, mt, nt, NT, b0, nks, acc_out);
      return;
    }
#pragma unroll 1
    for (int h = 0; h < NT; ++h) {
      const int ya = min(8 * (nt + h) + 2 * t, b - 1), yb = min(8 * (nt + h) + 2 * t + 1, b - 1);
      const unsigned char* yp = yt.base + b0 * yt.blk;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      for (int r = 0; r < 16 * nks; ++r) {
        const double x0 = tc_ld(z0 - ca * 128 + TcTile::off(blk0, r, ca));
        const double x1 = tc_ld(z1 - cc * 128 + TcTile::off(blk1, r, cc));
        const double u = tc_ld(yp + TcTile::off(yt.blk, r, ya)), v = tc_ld(yp + TcTile::off(yt.blk, r, yb));
        s0 = fma(x0, u, s0);
        s1 = fma(x0, v, s1);
        s2 = fma(x1, u, s2);
        s3 = fma(x1, v, s3);
      }
      double* ao = acc_out + h * 128;
      ao[lane] += s0;
      ao[32 + lane] += s1;
      ao[64 + lane] += s2;
      ao[96 + lane] += s3;
    }
    return;
  }
  const FxScale k0 = fx_scale(E0), k1 = fx_scale(E1);
  FxScale kb[NT];
#pragma unroll
  for (int h = 0; h < NT; ++h) kb[h] = fx_scale(Eb[h]);
  const FxMask km = fx_masks();
  const bool small = nks <= 2;
  float acc[NT][7][4], sizes[NT][4], init[4];
  fx_init(init, small);
  auto step = [&](int ks, auto first) {
    const unsigned char *pa = z0 + ks * blk0, *pc = z1 + ks * blk1;
    const double2 u0 = tc_ld2(pa + oa), u1 = tc_ld2(pa + (oa ^ 16));
    const double2 w0 = tc_ld2(pc + ob), w1 = tc_ld2(pc + (ob ^ 16));
    uint32_t bd[NT][7][2];
#pragma unroll
    for (int h = 0; h < NT; ++h) {
      const unsigned char* py = y0[h] + ks * yt.blk;
      const double2 v0 = tc_ld2(py + oy[h]), v1 = tc_ld2(py + (oy[h] ^ 16));
      FxPair q0 = fx_pair(v0.x, v0.y, kb[h], km), q1 = fx_pair(v1.x, v1.y, kb[h], km);
      fx_bdigits(q0, q1, bd[h], km);
    }
    FxPair p00 = fx_pair(u0.x, u0.y, k0, km), p01 = fx_pair(u1.x, u1.y, k0, km);
    FxPair p10 = fx_pair(w0.x, w0.y, k1, km), p11 = fx_pair(w1.x, w1.y, k1, km);
    fx_step<decltype(first)::value, NT>(acc, p00, p10, p01, p11, bd, km, init, GUARD ? sizes : nullptr);
  };
  step(0, FxTrue());
#pragma unroll 1
  for (int ks = 1; ks < nks; ++ks) step(ks, FxFalse());
  if constexpr (GUARD) {
    bool few = false;
#pragma unroll
    for (int h = 0; h < NT; ++h) {
      const bool f = tc_gram_small(sizes[h], nks, E0, E1, Eb[h]);  // (whole warp: shuffles)
      few = few || f;
    }
    if (__any_sync(0xffffffffu, few)) {
      tc_gram_fma(xt, yt, ax, zr, b, mt, nt, NT, b0, nks, acc_out);
      return;
    }
  }
#pragma unroll
  for (int h = 0; h < NT; ++h) tc_gram_flush(acc[h], small, E0, E1, Eb[h], zr - i0 > 8, acc_out + h * 128);
}

// The same for Y^T Y of at most 8 columns: the A digits are the B digits, and rows 8..15 of
// A hold the next digit, so that one product serves the pairs (I, J) and (I + 1, J): the
// sums of level l are acc[l][0, 1] + acc[l - 1][2, 3].
static __device__ __forceinline__ void tc_gram_sym8(const TcTile yt, int b, int b0, int nks, double* acc_out) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int yc = min(g, b - 1);
  const unsigned char* y0 = yt.base + b0 * yt.blk + yc * 128;
  const int oy = ((2 * t) ^ (yc & 7)) << 4;
  FxMax mb;
  for (int ks = 0; ks < nks; ++ks) {
    const unsigned char* py = y0 + ks * yt.blk;
    const double2 v0 = tc_ld2(py + oy), v1 = tc_ld2(py + (oy ^ 16));
    mb.add(v0.x, v0.y);
    mb.add(v1.x, v1.y);
  }
  mb.reduce4();
  const int Eb = mb.scale();
  if (__any_sync(0xffffffffu, Eb == 0)) {
    const int ya = min(2 * t, b - 1), yb = min(2 * t + 1, b - 1);
    const unsigned char* yp = yt.base + b0 * yt.blk;
    double s0 = 0.0, s1 = 0.0;
    for (int r = 0; r < 16 * nks; ++r) {
      const double x = tc_ld(yp + TcTile::off(yt.blk, r, yc));
      s0 = fma(x, tc_ld(yp + TcTile::off(yt.blk, r, ya)), s0);
      s1 = fma(x, tc_ld(yp + TcTile::off(yt.blk, r, yb)), s1);
    }
    acc_out[lane] += s0;
    acc_out[32 + lane] += s1;
    return;
  }
  const FxScale kb = fx_scale(Eb);
  const FxMask km = fx_masks();
  const bool small = nks <= 2;
  float acc[7][4], init[4];
  fx_init(init, small);
  auto step = [&](int ks, auto first) {
    const unsigned char* py = y0 + ks * yt.blk;
    const double2 v0 = tc_ld2(py + oy), v1 = tc_ld2(py + (oy ^ 16));
    uint32_t bd[7][2];
    FxPair q0 = fx_pair(v0.x, v0.y, kb, km), q1 = fx_pair(v1.x, v1.y, kb, km);
    fx_bdigits(q0, q1, bd, km);
#pragma unroll
    for (int I = 0; I < 7; I += 2) {
      const uint32_t a1 = I < 6 ? bd[I + 1][0] : 0u, a3 = I < 6 ? bd[I + 1][1] : 0u;
#pragma unroll
      for (int J = 0; J + I <= 6; ++J) {
        if (decltype(first)::value && I == 0)
          fx_mma_first(acc[J], bd[0][0], a1, bd[0][1], a3, bd[J][0], bd[J][1], init);
        else
          fx_mma(acc[I + J], bd[I][0], a1, bd[I][1], a3, bd[J][0], bd[J][1]);
      }
    }
  };
  step(0, FxTrue());
#pragma unroll 1
  for (int ks = 1; ks < nks; ++ks) step(ks, FxFalse());
  fx_ints(acc, small);
#pragma unroll
  for (int l = 6; l > 0; --l)
#pragma unroll
    for (int o = 0; o < 2; ++o)
      acc[l][o] = __int_as_float(__float_as_int(acc[l][o]) + __float_as_int(acc[l - 1][2 + o]));
  const int Ea = __shfl_sync(0xffffffffu, Eb, 8 * t), Ec = __shfl_sync(0xffffffffu, Eb, 8 * t + 4);
  acc_out[lane] = fma(fx_join(acc, 0), fx_weight(Eb, Ea), acc_out[lane]);
  acc_out[32 + lane] = fma(fx_join(acc, 1), fx_weight(Eb, Ec), acc_out[32 + lane]);
}

// Digits of the coefficients C (a x b, ld ldc, global) as B fragments of the update: for
// N tile nt and K step ks (KS = ceil(a / 16) of them), digit J at
// cf[((nt KS + ks) 7 + J) 32 + lane]; ec[c] the scale of column c (ceil(b / 8) * 8
// entries).  *bad is set when a column needs the float64 path.  Whole block; ends with a
// barrier.
static __device__ void tc_build_c(const double* C, int ldc, int a, int b, uint2* cf, int* ec, int* bad) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int KS = (a + 15) >> 4, NB = (b + 7) >> 3;
  const FxMask km = fx_masks();
  if (threadIdx.x == 0) *bad = 0;
  __syncthreads();
  for (int c = warp; c < 8 * NB; c += nw) {
    FxMax m;
    if (c < b)
      for (int k = lane; k < a; k += 32) m.add(C[k + (size_t)c * ldc], 0.0);
    m.m = __reduce_max_sync(0xffffffffu, m.m);
    m.nz = __reduce_or_sync(0xffffffffu, m.nz);
    const int E = m.scale();
    if (lane == 0) {
      ec[c] = E;
      if (E == 0) atomicOr(bad, 1);
    }
  }
  __syncthreads();
  for (int t0 = warp; t0 < NB * KS; t0 += nw) {
    const int ks = t0 % KS, nt = t0 / KS, g = lane >> 2, t = lane & 3;
    const int c = 8 * nt + g, k = 16 * ks + 2 * t;
    const FxScale key = fx_scale(max(ec[c], FX_EMIN));
    double v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int kk = k + (i & 1) + 8 * (i >> 1);
      v[i] = (kk < a && c < b) ? C[kk + (size_t)c * ldc] : 0.0;
    }
    FxPair q0 = fx_pair(v[0], v[1], key, km), q1 = fx_pair(v[2], v[3], key, km);
    uint32_t bd[7][2];
    fx_bdigits(q0, q1, bd, km);
#pragma unroll
    for (int J = 0; J < 7; ++J) cf[((size_t)t0 * 7 + J) * 32 + lane] = make_uint2(bd[J][0], bd[J][1]);
  }
  __syncthreads();
}

// digits of the NT column tiles from n0 at K step ks (the last tile stands in for one past it)
template <int NT>
static __device__ __forceinline__ void tc_load_b(const uint2* cf, int n0, int NB, int KS, int ks, int lane,
                                                 uint32_t (&bd)[NT][7][2]) {
#pragma unroll
  for (int h = 0; h < NT; ++h) {
    const uint2* q = cf + ((size_t)(min(n0 + h, NB - 1) * KS + ks) * 7) * 32 + lane;
#pragma unroll
    for (int J = 0; J < 7; ++J) {
      const uint2 u = q[J * 32];
      bd[h][J][0] = u.x;
      bd[h][J][1] = u.y;
    }
  }
}

// y -= x C for the 16 tile rows of one block (xb: a columns padded with zeros to a multiple
// of 16, yb: b columns, both block bases).  A row's scale is the largest exponent of its a entries.  Lane (g, t) owns rows
// g and g + 8, columns 2t, 2t+1, 2t+8, 2t+9 of every 16-column step.
// NT column tiles at a time share the digits of x.
template <int NT>
static __device__ __forceinline__ void tc_update_rows(const unsigned char* xb, unsigned char* yb, int a, int b,
                                                   const uint2* cf, const int* ec, int bad, const double* C,
                                                   int ldc) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int KS = (a + 15) >> 4, NB = (b + 7) >> 3, a8 = (a + 7) & ~7;
  // row g of columns 2t and 2t + 1; row g + 8 is 4 chunks (64 bytes) away
  const int o0 = 2 * t * 128 + (((g >> 1) ^ (2 * t)) << 4) + ((g & 1) << 3);
  const int o1 = (2 * t + 1) * 128 + (((g >> 1) ^ (2 * t + 1)) << 4) + ((g & 1) << 3);
  FxMax m0, m1;
  for (int k8 = 0; k8 < a8; k8 += 8) {
    const unsigned char* p = xb + k8 * 128;
    m0.add(tc_ld(p + o0), tc_ld(p + o1));
    m1.add(tc_ld(p + (o0 ^ 64)), tc_ld(p + (o1 ^ 64)));
  }
  m0.reduce4();
  m1.reduce4();
  const int E0 = m0.scale(), E1 = m1.scale();
  if (__any_sync(0xffffffffu, E0 == 0 || E1 == 0) || bad) {
    for (int e = lane; e < 16 * b; e += 32) {
      const int r = e & 15, c = e >> 4;
      double* yp = reinterpret_cast<double*>(yb + TcTile::off(0, r, c));
      double v = *yp;
      for (int i = 0; i < a; ++i) v = fma(-tc_ld(xb + TcTile::off(0, r, i)), C[i + (size_t)c * ldc], v);
      *yp = v;
    }
    return;
  }
  const FxScale k0 = fx_scale(E0), k1 = fx_scale(E1);
  const FxMask km = fx_masks();
  const bool small = KS <= 2;
  for (int n0 = 0; n0 < NB; n0 += NT) {
    float acc[NT][7][4], init[4];
    fx_init(init, small);
    auto step = [&](int ks, auto first) {
      const unsigned char* p = xb + ks * 2048;
      FxPair p00 = fx_pair(tc_ld(p + o0), tc_ld(p + o1), k0, km);
      FxPair p10 = fx_pair(tc_ld(p + (o0 ^ 64)), tc_ld(p + (o1 ^ 64)), k1, km);
      FxPair p01 = fx_pair(tc_ld(p + 1024 + o0), tc_ld(p + 1024 + o1), k0, km);
      FxPair p11 = fx_pair(tc_ld(p + 1024 + (o0 ^ 64)), tc_ld(p + 1024 + (o1 ^ 64)), k1, km);
      uint32_t bd[NT][7][2];
      tc_load_b<NT>(cf, n0, NB, KS, ks, lane, bd);
      fx_step<decltype(first)::value, NT>(acc, p00, p10, p01, p11, bd, km, init);
    };
    step(0, FxTrue());
#pragma unroll 1
    for (int ks = 1; ks < KS; ++ks) step(ks, FxFalse());
#pragma unroll
    for (int h = 0; h < NT; ++h) {
      const int nt = n0 + h;
      if (nt >= NB) break;
      fx_ints(acc[h], small);
      unsigned char* yt = yb + nt * 1024;
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        const int c = 8 * nt + 2 * t + (o & 1);
        const double v = fx_join(acc[h], o);
        if (c < b) {
          double* yp = reinterpret_cast<double*>(yt + (((o & 1) ? o1 : o0) ^ ((o >> 1) * 64)));
          *yp = fma(-v, fx_weight(o >> 1 ? E1 : E0, ec[c]), *yp);
        }
      }
    }
  }
}

// y = y Inv for the 16 tile rows of one block (yb: b columns padded with zeros to a multiple
// of 16), Inv upper triangular as B fragments (tc_build_c).  Pairs of column tiles are finished
// from the right: tiles nt, nt + 1 (nt even) read columns up to 8 nt + 15 only.
static __device__ __forceinline__ void tc_trmul_rows(unsigned char* yb, int b, const uint2* cf, const int* ec, int bad,
                                                     const double* Inv) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int KS = (b + 15) >> 4, NB = (b + 7) >> 3;
  const int o0 = 2 * t * 128 + (((g >> 1) ^ (2 * t)) << 4) + ((g & 1) << 3);
  const int o1 = (2 * t + 1) * 128 + (((g >> 1) ^ (2 * t + 1)) << 4) + ((g & 1) << 3);
  FxMax m0, m1;
  for (int k8 = 0; k8 < b; k8 += 8) {
    const unsigned char* p = yb + k8 * 128;
    m0.add(tc_ld(p + o0), tc_ld(p + o1));
    m1.add(tc_ld(p + (o0 ^ 64)), tc_ld(p + (o1 ^ 64)));
  }
  m0.reduce4();
  m1.reduce4();
  const int E0 = m0.scale(), E1 = m1.scale();
  if (__any_sync(0xffffffffu, E0 == 0 || E1 == 0) || bad) {
    if (lane < 16)
      for (int c = b - 1; c >= 0; --c) {
        double v = 0.0;
        for (int i = 0; i <= c; ++i) v = fma(tc_ld(yb + TcTile::off(0, lane, i)), Inv[i + (size_t)c * b], v);
        *reinterpret_cast<double*>(yb + TcTile::off(0, lane, c)) = v;
      }
    return;
  }
  const FxScale k0 = fx_scale(E0), k1 = fx_scale(E1);
  const FxMask km = fx_masks();
  for (int n0 = (NB - 1) & ~1; n0 >= 0; n0 -= 2) {
    const int ks_end = (n0 >> 1) + 1;
    const bool small = ks_end <= 2;
    float acc[2][7][4], init[4];
    fx_init(init, small);
    auto step = [&](int ks, auto first) {
      const unsigned char* p = yb + ks * 2048;
      FxPair p00 = fx_pair(tc_ld(p + o0), tc_ld(p + o1), k0, km);
      FxPair p10 = fx_pair(tc_ld(p + (o0 ^ 64)), tc_ld(p + (o1 ^ 64)), k1, km);
      FxPair p01 = fx_pair(tc_ld(p + 1024 + o0), tc_ld(p + 1024 + o1), k0, km);
      FxPair p11 = fx_pair(tc_ld(p + 1024 + (o0 ^ 64)), tc_ld(p + 1024 + (o1 ^ 64)), k1, km);
      uint32_t bd[2][7][2];
      tc_load_b<2>(cf, n0, NB, KS, ks, lane, bd);
      fx_step<decltype(first)::value, 2>(acc, p00, p10, p01, p11, bd, km, init);
    };
    step(0, FxTrue());
#pragma unroll 1
    for (int ks = 1; ks < ks_end; ++ks) step(ks, FxFalse());
    __syncwarp();  // every lane has read these tiles' columns
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int nt = n0 + h;
      if (nt >= NB) break;
      fx_ints(acc[h], small);
      unsigned char* yt = yb + nt * 1024;
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        const int c = 8 * nt + 2 * t + (o & 1);
        const double v = fx_join(acc[h], o);
        if (c < b)
          *reinterpret_cast<double*>(yt + (((o & 1) ? o1 : o0) ^ ((o >> 1) * 64))) =
              v * fx_weight(o >> 1 ? E1 : E0, ec[c]);
      }
    }
  }
}

}  // namespace rbo
