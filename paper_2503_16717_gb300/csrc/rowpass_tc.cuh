// The float64 row pass with its contractions on the fp16 tensor cores.
//
// y' = (y - x C) Tri^-1 per row, written back, and over the rows Z = [x, y']^T y' or the
// sparse sketch S y' (see rowpass.cu for the passes).  The projection and the Gram run on
// exact fixed-point digits (tc_fixed.cuh, tc_tile.cuh) instead of the float64 pipe, which
// bound those passes at 15-20 % of the HBM rate; triangular solves stay float64.
//
// CTAs of 4 warps, several per SM: tiles of T rows come in as tensor copies of 16-row
// boxes (one thread issues a handful per tile), double buffered; rows past n read as zero.
// Arrays a tensor copy cannot address (odd leading dimension, unaligned base, 2^31 rows) come in
// by asynchronous copies of 8 bytes that all threads issue, into the same stages at the same
// places (n = 400001 at an odd leading dimension: Gram call of 64 x 5 columns 187 us, one-stage of
// 61 columns 6.1 ms; plain loads in front of each tile 501 us and 10.2 ms).  Per tile
//   A  every warp updates its own 16-row blocks; triangular solve, one row per thread in
//      registers; write-back;
//   S  (sketch passes) the y' of the tile as 54-bit integers on one scale per column, and
//      their signed sums per sketch row from the tile's schedule record: the thread that
//      owns a slot of the record sums the slot's entries and adds them to the row's 64-bit
//      integer accumulators.  A column's scale rises when a value is past it, and the accumulators
//      with it.  They enter the CTA's float64 partial before a sketch row can have summed 384
//      entries (a few thousand rows, by the tiles' largest counts), so that most tiles cost no
//      float64 operation per sketch row.  Where the sketch itself is the result, the scale also
//      falls when a tile's values are all 2^SK_FAR below it, and the accumulators enter the partial
//      when it falls or rises by more than SK_RISE: a value is then off by at most
//      2^(SK_FAR - 1 + SK_RISE - 54) of the largest of its own tile.  (In the orthogonalization,
//      whose errors are measured against the norms of the columns, that would cost 26 % of the pass
//      on a basis whose sizes vary over the grid: convection-diffusion 2048^2.)
//   B  the Gram items, (16 Z columns) x (8 Y' columns) x (a chunk of kc rows), are dealt
//      to the warps; an item always goes to the same warp, which keeps its float64 sums
//      in its own shared-memory slots.
// Measured on GB300, n = 2^22, b = 5, mean over a = 1, 6, .. 56 (float64-pipe kernels it
// replaces -> here): Gram 1116 -> 468 us, update + Gram 1337 -> 539 us, solve + Gram
// 1345 -> 549 us, update + sketch (d = 244, 8 entries a row) 1521 -> 747 us; orthogonalization
// of 61 columns in one stage 72.5 -> 33.6 ms, in two 76.3 -> 32.7 ms.  The integer conversion
// bounds it (IPC 2.2 of 4, ALU pipe 45-50 %, tensor pipe 30 %, DRAM 35 % of the copy rate; a
// pass of one to 16 columns X costs the same), in the sketch passes the bank conflicts of the
// gathered sums too (870 shared-memory cycles a 64-row tile, 313 without conflicts).
// The last CTAs reduce the partials in a fixed order and run the small dense epilogue
// (rowpass_common.cuh).
#pragma once

#include <cuda.h>

#include <algorithm>

#include "rowpass_common.cuh"
#include "tc_tile.cuh"
#include "tma_map.cuh"

namespace rbo {

constexpr int TC_NT = 128;
constexpr int TC_NW = TC_NT / 32;
constexpr int SK_FAR = 6;   // sketch scales: 16 rows of like values nearly never lie all below 2^-6
constexpr int SK_RISE = 3;  // of the largest seen; a scale with room of one bit rises by 2 at least

struct TcDev {
  CUtensorMap tmX, tmY;
  PassDev P;
};

// Panels of more than 8 columns after the inverse or an update alone (wide): two column tiles
// at a time, which share the digits of the left operand (2^22 rows, a = 31, b = 30: inverse +
// Gram 2374 -> 1990 us, update + Gram 2675 -> 2150 us, inverse alone 1034 -> 958 us).
__host__ __device__ constexpr bool tc_wide(int tri, int g) { return tri == 2 || g == 3; }
// CTAs per SM the registers are bounded for: the substitution alone waits for the float64 pipe
// and wants warps (2^22 rows, b = 5: 153 us at 4, 138 at 8 with spills, 135 at 6); with the
// Gram of 8 columns 5 (251 -> 246 us); with a general Gram 3, free of spills, since the shared
// memory allows few more (solve + Gram 572 -> 549 us, update + solve + Gram 822 -> 781 us);
// the wide ones need 168 registers; everything else 128.
constexpr int tc_min_ctas(bool hc, int tri, int g) {
  if (tc_wide(tri, g) || (tri == 1 && g == 1)) return 3;
  return tri == 1 && !hc ? (g == 0 ? 6 : (g == 2 ? 5 : 4)) : 4;
}

// Asynchronous copies of a tile by all threads: `left` rows of src from the tile's first one on,
// cols columns, into blocks of 16 rows, zeros past them; bytes is a multiple of 16.  Not inlined:
// the kernels' own code stays as short as without them.
static __device__ __noinline__ void tc_copy_cols(unsigned char* dst, int blk, const double* src, int64_t ld, int cols,
                                                 int tsh, int64_t left) {
  for (int t = threadIdx.x; t < cols << tsh; t += TC_NT) {
    const int c = t >> tsh, r = t & ((1 << tsh) - 1);
    const bool in = r < left;
    cp_async8(dst + TcTile::off(blk, r, c), in ? src + c * ld + r : src, in);
  }
}
static __device__ __noinline__ void tc_copy_bytes(unsigned char* dst, const uint8_t* src, int bytes) {
  for (int t = 16 * threadIdx.x; t < bytes; t += 16 * TC_NT) cp_async16(dst + t, src + t);
}

// Sketch sums into the CTA's partial (= for the first time, then +=), each thread its own entries;
// the sums start again from zero
static __device__ __forceinline__ void sk_flush(long long* ska, int d, int b, const int* scale, const bool* nan,
                                                double* part, bool first, bool mixed) {
  for (int t = threadIdx.x; t < d * b; t += TC_NT) {
    const int c = t / d;
    if (mixed) {
      part[t] = (double)reinterpret_cast<const float*>(ska)[t];
      continue;
    }
    const int sc = scale[c];
    double v = (double)ska[t];
    v = sc >= 60 ? v * __hiloint2double((sc - 53) << 20, 0) : scalbn(v, sc - 1076);
    if (nan[c]) v = __longlong_as_double(0x7FF8000000000000LL);
    part[t] = first ? v : part[t] + v;
    ska[t] = 0;
  }
}
struct SkScales {   // per column:
  int scale[64];    // exponent field of the scale,
  short base[64];   // of the scale at the last flush,
  short now[64];    // of the next scale
  bool nan[64];     // the column has a value that is not finite
  int rescale;      // set when a warp found a value past its scale, or 16 far below it
};
// Scales for this tile (y' at ys, bytes from the start of the dynamic shared memory, as ska and
// skf) and its values on them; true when the sums (cnt: entries a row can hold) went into the
// partial.  Whole block, all threads past the conversion of the tile; ends with a barrier.  Not
// inlined: it runs every few dozen tiles, and a pass with it in its loop takes 5 % longer.
static __device__ __noinline__ bool sk_rescale(SkScales& S, int ys, int yblk, int tsh, int d, int b, int ska_off,
                                               int skf_off, double* part, bool first, bool full, int cnt,
                                               bool follow) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  long long *ska = reinterpret_cast<long long*>(smem_raw + ska_off), *skf = reinterpret_cast<long long*>(smem_raw + skf_off);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = 1 << tsh;
  bool change = false, flush = full;
  if (S.rescale != 0) {
    for (int c = warp; c < b; c += TC_NW) {
      int ex = 0;
      for (int r = lane; r < T; r += 32)
        ex = max(ex, (__double2hiint(tc_ld(smem_raw + ys + TcTile::off(yblk, r, c))) >> 20) & 0x7FF);
      ex = __reduce_max_sync(0xffffffffu, ex);
      if (lane == 0) {
        // (room to grow, but never up to the exponent field of Inf and NaN, which must stay past
        // every scale)
        const int old = S.scale[c];
        if (ex == 0x7FF) S.nan[c] = true;
        S.now[c] = (short)(ex != 0x7FF && ex > 0 && (ex > old || (follow && ex + SK_FAR <= old)) ? min(ex + 1, 0x7FE) : old);
      }
    }
    __syncthreads();
    for (int c = lane; c < b; c += 32) {
      const int old = S.scale[c], now = S.now[c];
      change = change || now != old;
      flush = flush || now < old || (follow && old > 0 && now > S.base[c] + SK_RISE);
    }
    change = __any_sync(0xffffffffu, change);  // (the same in every warp)
    flush = __any_sync(0xffffffffu, flush) && cnt > 0;
  }
  if (flush) {  // sums on the scales they were formed with
    sk_flush(ska, d, b, S.scale, S.nan, part, first, false);
  } else if (change && cnt > 0) {  // rises without a flush: the sums move along
    for (int t = tid; t < d * b; t += TC_NT) {
      const int k = S.now[t / d] - S.scale[t / d];
      if (k > 0 && ska[t] != 0) ska[t] = k >= 62 ? 0 : (ska[t] + (1LL << (k - 1))) >> k;
    }
  }
  __syncthreads();  // scales read above
  if (tid < b) {
    if (change) S.scale[tid] = S.now[tid];
    if (flush || cnt == 0 || S.base[tid] == 0) S.base[tid] = (short)S.scale[tid];
  }
  if (tid == 0) S.rescale = 0;
  if (change) {
    __syncthreads();
    for (int t = tid; t < T * b; t += TC_NT) {
      const int c = t >> tsh, r = t & (T - 1);
      const double v = tc_ld(smem_raw + ys + TcTile::off(yblk, r, c));
      const long long f = S.nan[c] ? 0 : fx_round54(v, S.scale[c]);
      skf[2 * r * b + c] = f;
      skf[(2 * r + 1) * b + c] = -f;
    }
  }
  __syncthreads();
  return flush;
}

// HC: projection (C digits); TRI: triangular factor, 0 none, 1 substitution, 2 product with its
// inverse (digits); G: Gram, 0 none, 1 general, 2 of at most
// 8 columns of Y' alone, 3 of more columns of Y' alone after an update, 4 general with a bound for
// every entry; SK: sparse sketch (no triangle, no Gram).  Each kind of pass is its
// own kernel: fewer live registers and less code than one kernel with all phases.
template <bool HC, int TRI, int G, bool SK>
__global__ void __launch_bounds__(TC_NT, tc_min_ctas(HC, TRI, G)) rowpass_tc_kernel(const __grid_constant__ TcDev D) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // X is read by the update alone when the pass has no general Gram: one X stage then, its
  // next tile copied in once every warp has updated its rows (Y keeps two stages), which
  // leaves room for four CTAs per SM.  With a triangle and a general Gram (XL) X is read by
  // the Gram alone and comes in while the panel's rows are solved: one stage again, and tiles
  // of 128 rows in the same shared memory, whose four warps each have 32 rows to solve (64
  // rows: two warps idle, 2^22 x 61: 742 -> 674 us; b = 30 with the inverse 2683 -> 2393 us).
  constexpr bool HT = TRI != 0, inv = TRI == 2;
  constexpr bool XL = HT && !HC && G == 1, XS = (HC && G != 1) || XL;
  // panels of more than 8 columns: two column tiles at a time
  constexpr int NT = tc_wide(TRI, G) ? 2 : 1;
  __shared__ __align__(8) uint64_t bars[NST], barx;
  __shared__ int s_flag;
  __shared__ int s_last;
  __shared__ int s_bad;
  __shared__ SkScales s_sk;  // sketch
  const PassDev& P = D.P;
  const RowPass& rp = P.p;
  if (read_code(P.status) != 0) return;
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int T = P.T, tsh = 31 - __clz(T), a = rp.a, b = rp.b;
  const int ax = rp.acc_x ? a : 0;
  const int64_t n = rp.n;
  const int xblk = P.xblk, yblk = P.yblk, nblk16 = T >> 4;
  double* Ts = reinterpret_cast<double*>(smem + P.off_tri);
  double* dinv = reinterpret_cast<double*>(smem + P.off_dinv);
  uint2* cf = reinterpret_cast<uint2*>(smem + P.off_c);
  int* ec = reinterpret_cast<int*>(smem + P.off_ec);
  double* accs = reinterpret_cast<double*>(smem + P.off_acc);
  const int ldc = rp.ldc > 0 ? rp.ldc : a;
  const int d = SK ? rp.sk_d : 0;            // scattered sketch rows
  long long* ska = reinterpret_cast<long long*>(smem + P.off_sk);   // d x b sums
  long long* skf = reinterpret_cast<long long*>(smem + P.off_skf);  // T x 2 x b tile values
  const int rec_n = d > 0 ? rp.sk.rec_bytes : 0;

  if (tid == 0) {
    for (int s = 0; s < NST; ++s) mbar_init(&bars[s], 1);
    mbar_init(&barx, 1);
    fence_mbar_init();
  }
  __syncthreads();

  auto stage_X = [&](int s) { return smem + (XS ? 0 : (size_t)s * P.stage_bytes); };
  auto stage_Y = [&](int s) { return smem + (size_t)nblk16 * xblk + (size_t)s * P.stage_bytes; };
  auto stage_R = [&](int s) { return stage_Y(s) + (size_t)nblk16 * yblk; };
  // one thread copies a tile into stage s
  auto issue_tile = [&](int tile, int s) {
    const int r0 = tile * T;
    mbar_arrive_expect_tx(&bars[s], (uint32_t)(T * 8) * (uint32_t)((XS ? 0 : a) + b) + (uint32_t)rec_n);
    if (d > 0) bulk_copy_g2s(stage_R(s), rp.sk.rec + (size_t)tile * rec_n, (uint32_t)rec_n, &bars[s]);
    for (int k = 0; k < nblk16; ++k) {
      if (!XS && a > 0) tma_load_rows(stage_X(s) + k * xblk, &D.tmX, r0 + 16 * k, &bars[s]);
      tma_load_rows(stage_Y(s) + k * yblk, &D.tmY, r0 + 16 * k, &bars[s]);
    }
  };
  auto issue_x = [&](int tile) {  // XS: the tile's X alone
    mbar_arrive_expect_tx(&barx, (uint32_t)(T * 8) * (uint32_t)a);
    if (a > 0)
      for (int k = 0; k < nblk16; ++k) tma_load_rows(smem + k * xblk, &D.tmX, tile * T + 16 * k, &barx);
  };

  // the same without the copy engine, by all threads; a group per call
  auto copy_tile = [&](int tile, int s) {
    const int64_t r0 = (int64_t)tile * T;
    if (!XS) tc_copy_cols(stage_X(s), xblk, rp.X + r0, rp.ldx, a, tsh, n - r0);
    tc_copy_cols(stage_Y(s), yblk, rp.Y + r0, rp.ldy, b, tsh, n - r0);
    if (rec_n > 0) tc_copy_bytes(stage_R(s), rp.sk.rec + (size_t)tile * rec_n, rec_n);
    cp_async_commit();
  };
  auto copy_x = [&](int tile) {
    const int64_t r0 = (int64_t)tile * T;
    tc_copy_cols(smem, xblk, rp.X + r0, rp.ldx, a, tsh, n - r0);
    cp_async_commit();
  };

  // XS: X of a later tile once every warp is done with the one before it
  auto next_x = [&](int tile) {
    if (tile >= P.ntiles) return;
    if (!P.use_bulk) {
      copy_x(tile);
    } else if (tid == 0) {
      fence_proxy_async();
      issue_x(tile);
    }
  };

  // the first tile is in flight while the small matrices are prepared
  uint32_t phx = 0u;  // (a stage's phase: the parity of the tiles it held)
  const int first = blockIdx.x;
  if (first < P.ntiles) {
    if (!P.use_bulk) {
      copy_tile(first, 0);
      if (XS) copy_x(first);
    } else if (tid == 0) {
      issue_tile(first, 0);
      if (XS) issue_x(first);
    }
  }
  // the padding columns of every block hold zeros (the copies do not touch them)
  for (int s = 0; s < NST; ++s) {
    const int pa = (xblk >> 7) - a, pb = (yblk >> 7) - b;
    for (int t = tid; t < nblk16 * (pa + pb) * 8; t += TC_NT) {
      const int k = t / ((pa + pb) * 8), u = t - k * (pa + pb) * 8, c = u >> 3;
      if (XS && s > 0 && c < pa) continue;  // (the first X tile is in flight around its padding)
      unsigned char* p = c < pa ? stage_X(s) + k * xblk + (a + c) * 128 : stage_Y(s) + k * yblk + (b + c - pa) * 128;
      *reinterpret_cast<uint4*>(p + 16 * (u & 7)) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  if (HT && !inv) {
    const int ldt = rp.ldtri > 0 ? rp.ldtri : b;
    for (int t = tid; t < b * b; t += TC_NT) {
      const int i = t % b, c = t / b;
      Ts[t] = (i <= c) ? rp.Tri[i + (size_t)c * ldt] : 0.0;
    }
    for (int t = tid; t < b; t += TC_NT) dinv[t] = 1.0 / rp.Tri[t + (size_t)t * ldt];
  }
  if constexpr (G != 0)
    for (int t = tid; t < P.items * 128 * NT; t += TC_NT) accs[t] = 0.0;
  if constexpr (SK) {
    for (int t = tid; t < d * b; t += TC_NT) ska[t] = 0;  // (all-zero bits also as float32 pairs)
    if (tid < 64) {
      s_sk.scale[tid] = s_sk.base[tid] = 0;
      s_sk.nan[tid] = false;
    }
    if (tid == 0) s_sk.rescale = 0;
  }
  if (HC && P.c_digits) tc_build_c(rp.C, ldc, a, b, cf, ec, &s_bad);
  if (inv) tc_build_c(rp.Inv, b, b, b, cf, ec, &s_bad);
  __syncthreads();
  const int bad_c = HC ? (P.c_digits ? s_bad : 1) : (inv ? s_bad : 0);
  // rows of a tile a warp owns from the update to the sums of a chunk: rpw from rw
  const int rsh = max(4, tsh - 2), rpw = 1 << rsh, rw = warp * rpw, re = min(rw + rpw, T);
  double* mypart = P.L > 0 ? P.partials + (size_t)blockIdx.x * P.L : nullptr;
  const bool mixed = SK && rp.mixed;  // float32 values and sums of the sketch
  bool sk_first = true;  // nothing in the partial yet
  int sk_cnt = 0;  // entries a sketch row can have summed since the last flush
  const int q = P.blk_start[P.nblk];  // Gram items per chunk

  int it = 0;
  for (int tile = first; tile < P.ntiles; tile += gridDim.x, ++it) {
    const int s = it & 1;
    const int64_t r0 = (int64_t)tile * T;
    const int rows = (n - r0 < (int64_t)T) ? (int)(n - r0) : T;
    unsigned char* xs = stage_X(s);
    unsigned char* ys = stage_Y(s);
    if (P.use_bulk) {
      bool ok = mbar_wait_bounded(&bars[s], (uint32_t)(it >> 1) & 1u);
      if (XS && !XL) ok = mbar_wait_bounded(&barx, phx) && ok;
      if (__syncthreads_or(!ok)) {
        if (tid == 0) {
          set_error(P.status, RBO_ERR_TIMEOUT, 1);
          if (XL && it == 0) mbar_wait_bounded(&barx, phx);  // the other copy in flight
        }
        return;
      }
      if (!XL) phx ^= 1u;
      // prefetch the next tile into the other stage (its readers passed the barrier)
      const int nxt = tile + gridDim.x;
      if (tid == 0) {
        fence_proxy_async();
        if (XL && it > 0) issue_x(tile);
        if (nxt < P.ntiles) issue_tile(nxt, s ^ 1);
      }
    } else {
      cp_async_wait<0>();
      __syncthreads();  // the tile is in, the previous tile's readers are done
      const int nxt = tile + gridDim.x;
      if (XL && it > 0) copy_x(tile);
      if (nxt < P.ntiles) copy_tile(nxt, s ^ 1);
      else cp_async_commit();  // (an empty group: the waits below count groups)
    }

    // ---- A: y' in place in the Y stage -------------------------------------------
    // Each warp works on its own rows, without a block barrier.  Triangular solve: one row
    // per lane, column blocks of 8 in registers; each entry subtracts its terms in column
    // order, as an unblocked row-by-row substitution would.
    bool synced = false;  // the last step ended with a block barrier
    auto tri_solve = [&]() {
      if constexpr (inv) {
        for (int k = rw >> 4; k < re >> 4; ++k) tc_trmul_rows(ys + k * yblk, b, cf, ec, bad_c, rp.Inv);
        __syncwarp();
        return;
      }
      // (a warp with fewer than 32 rows would leave lanes idle: rows over the block then)
      const bool own = rpw >= 32;
      if (!own && HC) __syncthreads();
      for (int r = own ? rw + lane : tid; r < (own ? re : T); r += own ? 32 : TC_NT) {
        for (int c0 = 0; c0 < b; c0 += 8) {
          const int cw = min(8, b - c0);
          double v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (j < cw) v[j] = tc_ld(ys + TcTile::off(yblk, r, c0 + j));
          for (int i = 0; i < c0; ++i) {
            const double yi = -tc_ld(ys + TcTile::off(yblk, r, i));
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (j < cw) v[j] = fma(yi, Ts[i + (c0 + j) * b], v[j]);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (j < cw) {
#pragma unroll
              for (int i = 0; i < j; ++i) v[j] = fma(-v[i], Ts[c0 + i + (c0 + j) * b], v[j]);
              v[j] *= dinv[c0 + j];
              *reinterpret_cast<double*>(ys + TcTile::off(yblk, r, c0 + j)) = v[j];
            }
        }
      }
      if (own) __syncwarp();
      else __syncthreads();
      synced = !own;
    };
    if constexpr (HC) {
      for (int k = rw >> 4; k < re >> 4; ++k)
        tc_update_rows<NT>(xs + k * xblk, ys + k * yblk, a, b, cf, ec, bad_c, rp.C, ldc);
      synced = false;
      if (XS && !SK) {
        __syncthreads();  // every warp is done with X (sketch passes: at their own barrier)
        synced = true;
        next_x(tile + gridDim.x);
      } else {
        __syncwarp();
      }
    }
    if (HT) tri_solve();
    if (rp.write_y) {
      if (P.use_bulk) {  // two rows per lane
        const int h = (re - rw) >> 1, hsh = 31 - __clz(max(h, 1));
        for (int t = lane; t < b * h; t += 32) {
          const int c = t >> hsh, r = rw + (t & (h - 1)) * 2;
          const double2 v = tc_ld2(ys + TcTile::off(yblk, r, c));
          double* dst = rp.Y + c * rp.ldy + r0 + r;
          if (r + 1 < rows)
            *reinterpret_cast<double2*>(dst) = v;
          else if (r < rows)
            *dst = v.x;
        }
      } else {
        for (int c = 0; c < b; ++c)
          for (int r = rw + lane; r < min(re, rows); r += 32)
            rp.Y[c * rp.ldy + r0 + r] = tc_ld(ys + TcTile::off(yblk, r, c));
      }
    }

    // ---- S: sketch sums ---------------------------------------------------------------
    if constexpr (SK) {
      // Every warp converts its 16 rows with the columns' current scales, two columns at a time;
      // only a tile with a value past a scale (or not finite), or with 16 rows of a column all
      // far below it, takes the block-wide path below.
      bool past = false, low = false;
      for (int t0 = 0; t0 < (re - rw) * b; t0 += 32) {
        const int t = t0 + lane, r = rw + (t & 15), c = t >> 4;
        const bool in = c < b;
        const double v = in ? tc_ld(ys + TcTile::off(yblk, r, c)) : 0.0;
        if (mixed) {
          if (in) {
            const float f = f64_to_f32_int(v);
            reinterpret_cast<float*>(skf)[2 * r * b + c] = f;
            reinterpret_cast<float*>(skf)[(2 * r + 1) * b + c] = -f;
          }
        } else {
          const int sc = in ? s_sk.scale[c] : 0, ex = (__double2hiint(v) >> 20) & 0x7FF;
          past = past || ex > sc;
          const unsigned near = rp.elementwise ? __ballot_sync(0xffffffffu, ex + SK_FAR > sc) : 0xffffffffu;
          if (near < 0x10000u || (near & 0xFFFFu) == 0u) {
            const unsigned some = __ballot_sync(0xffffffffu, ex > 0);
            low = low || (near < 0x10000u && some >= 0x10000u) || ((near & 0xFFFFu) == 0u && (some & 0xFFFFu) != 0u);
          }
          if (in) {
            const long long f = fx_round54(v, sc);
            skf[2 * r * b + c] = f;
            skf[(2 * r + 1) * b + c] = -f;
          }
        }
      }
      if ((__any_sync(0xffffffffu, past) || low) && lane == 0) s_sk.rescale = 1;
      __syncthreads();
      if (XS) next_x(tile + gridDim.x);
      if (!mixed) {
        // the record's first slot has the tile's most entries in one sketch row
        const uint32_t m0 = *reinterpret_cast<const uint32_t*>(stage_R(s));
        const int most = m0 == 0xFFFFFFFFu ? 0 : (int)(m0 >> 23);
        const bool full = sk_cnt + most > 384;  // 2^54 * 384 < 2^63
        if (full || s_sk.rescale != 0) {
          const int base = (int)(smem - smem_raw);
          if (sk_rescale(s_sk, (int)(ys - smem_raw), yblk, tsh, d, b, base + P.off_sk, base + P.off_skf, mypart, sk_first,
                         full, sk_cnt, rp.elementwise != 0)) {
            sk_first = false;
            sk_cnt = 0;
          }
        }
        sk_cnt += most;
      }
      const uint32_t* meta = reinterpret_cast<const uint32_t*>(stage_R(s));
      for (int c0 = 0; c0 < b; c0 += CB) {
        const int cw = min(CB, b - c0);
        if (mixed) {
          RBO_CW_DISPATCH(sketch_tile_sums, cw, meta, rp.sk.mcap, reinterpret_cast<float*>(ska) + (size_t)c0 * d, d,
                          reinterpret_cast<const float*>(skf) + c0, b)
        } else {
          RBO_CW_DISPATCH(sketch_tile_sums, cw, meta, rp.sk.mcap, ska + (size_t)c0 * d, d, skf + c0, b)
        }
      }
    }

    // ---- B: Z += [x, y']^T y' ------------------------------------------------------
    if constexpr (G != 0) {
      // the chunks of sym8 items are the warps' own rows; general items read other warps'
      if (XL && P.use_bulk) {
        if (__syncthreads_or(!mbar_wait_bounded(&barx, phx))) {
          if (tid == 0) {
            set_error(P.status, RBO_ERR_TIMEOUT, 1);
            if (tile + (int)gridDim.x < P.ntiles) mbar_wait_bounded(&bars[s ^ 1], (uint32_t)((it + 1) >> 1) & 1u);
          }
          return;
        }
        phx ^= 1u;
      } else if (XL) {
        cp_async_wait<1>();  // X; the next tile's group came after it
        __syncthreads();
      } else if ((G == 1 || G == 3) && (HC || HT) && !synced) {
        __syncthreads();
      }
      const TcTile xt{xs, xblk}, yt{ys, yblk};
      for (int item = warp; item < P.items; item += TC_NW) {
        if constexpr (G == 2) {
          tc_gram_sym8(yt, b, (item * P.kc) >> 4, P.kc >> 4, accs + item * 128);
        } else {
          const int chunk = item / q, task = item - chunk * q;
          int nt = 0;
          while (nt + 1 < P.nblk && task >= P.blk_start[nt + 1]) ++nt;
          tc_gram_item<NT, G == 4>(xt, yt, ax, P.zr, b, task - P.blk_start[nt], nt * NT, (chunk * P.kc) >> 4, P.kc >> 4,
                           accs + item * 128 * NT);
        }
      }
    }
  }

  // ---------------- partials + fixed-order two-level tree -------------------------
  if (P.L == 0) return;
  __syncthreads();
  if constexpr (SK) sk_flush(ska, d, b, s_sk.scale, s_sk.nan, mypart, sk_first, mixed);
  if constexpr (G != 0)
  for (int o = tid; o < P.no; o += TC_NT) {
    const int i = o / b, c = o % b;
    // the entries of Y'^T Y' below the diagonal come from the upper triangle (the same
    // integer sums)
    int zi = i, zc = c;
    if (i >= ax && i - ax > c) {
      zi = ax + c;
      zc = i - ax;
    }
    const int task = P.blk_start[(zc >> 3) / NT] + (zi >> 4);
    const int ri = zi & 15, ci = zc & 7;
    const double* p = accs + (size_t)(task * NT + (zc >> 3) % NT) * 128 + (2 * (ri >> 3) + (ci & 1)) * 32 + 4 * (ri & 7) + (ci >> 1);
    double sum = 0.0;
    for (int item = 0; item < P.items; item += q) sum += p[(size_t)item * 128 * NT];
    mypart[o] = sum;
  }
  tree_reduce_epilogue(P, smem_raw, &s_flag, &s_last);
}

// The kernel of a kind of pass; null for a combination no pass uses
typedef void (*TcKernel)(TcDev);
TcKernel tc_kernel_g0(bool hc, int tri, bool sk);  // no Gram   (rowpass_tc_g0.cu)
TcKernel tc_kernel_g1(bool hc, int tri);            // general   (rowpass_tc_g1.cu)
TcKernel tc_kernel_g3();                            // wide Y'^T Y' after an update (rowpass_tc_g1.cu)
TcKernel tc_kernel_g4();                            // general with a bound for every entry (rowpass_tc_g1.cu)
TcKernel tc_kernel_g2(bool hc, int tri);            // Y'^T Y', at most 8 columns (rowpass_tc_g2.cu)

}  // namespace rbo
