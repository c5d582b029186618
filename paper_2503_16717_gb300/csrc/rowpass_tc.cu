// Launcher of the tensor-core row passes (kernels: rowpass_tc.cuh)
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "rowpass_tc.cuh"

namespace rbo {

// ------------------------------------------------------------------------------------
// launcher
// ------------------------------------------------------------------------------------
constexpr int TC_MAX_DEV = 64;
static std::mutex g_tc_mu;
static std::map<const void*, int> g_tc_smem[TC_MAX_DEV];  // kernel -> dynamic shared memory limit

int make_tensor_map(CUtensorMap* m, const double* base, int64_t n, int cols, int64_t ld) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_tc_mu);
    if (encode == nullptr) {
      void* fn = nullptr;
      cudaDriverEntryPointQueryResult q;
      if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
              cudaSuccess ||
          q != cudaDriverEntryPointSuccess || fn == nullptr) {
        cudaGetLastError();
        return RBO_ERR_CUDA;
      }
      encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
  }
  const cuuint64_t dims[2] = {(cuuint64_t)n, (cuuint64_t)cols};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 8};
  const cuuint32_t box[2] = {16u, (cuuint32_t)cols};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<double*>(base), dims,
                            strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? RBO_OK : RBO_ERR_CUDA;
}

static int tc_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= TC_MAX_DEV) dev = 0;
  return dev;
}

// Largest dynamic shared memory of a kernel; raises its limit to that on first use
static int tc_smem_limit(const void* kern) {
  const int dev = tc_device();
  std::lock_guard<std::mutex> lk(g_tc_mu);
  int& lim = g_tc_smem[dev][kern];
  if (lim == 0) {
    int optin = 0;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    size_t stat = 0;
    if (cudaFuncGetAttributes(&fa, kern) == cudaSuccess) stat = fa.sharedSizeBytes;
    lim = optin - (int)stat - 64;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, lim) != cudaSuccess) {
      cudaGetLastError();
      lim = 48 * 1024 - (int)stat;
    }
  }
  return lim;
}

// Shared memory of the streaming loop
struct TcLayout {
  int xblk, yblk;
  size_t stage_bytes, off_c, off_acc, off_tri, off_dinv, off_ec, off_sk, off_skf, bytes;
};
// digits: B fragments of C (or, inv, of the inverse of Tri) are held in shared memory
static TcLayout tc_layout(int a, int b, int T, int items, bool has_c, bool digits, bool has_tri, bool inv, int d,
                          int rec, bool xs) {
  TcLayout l;
  l.xblk = tc_blk_bytes(a, has_c ? 16 : 8);
  l.yblk = tc_blk_bytes(b, inv ? 16 : 8);
  // per stage: X, Y, record; with one X stage (xs) X comes first and a stage is Y and record
  const size_t xb = (size_t)(T / 16) * l.xblk;
  l.stage_bytes = (((size_t)(T / 16) * l.yblk + (xs ? 0 : xb) + rec) + 1023) & ~size_t(1023);
  size_t o = NST * l.stage_bytes + (xs ? xb : 0);
  const int NB = (b + 7) / 8, KS = ((inv ? b : a) + 15) / 16;
  l.off_c = o; o += digits ? (size_t)NB * KS * 7 * 256 : 0;
  l.off_acc = o; o += (size_t)items * 1024;
  l.off_sk = o; o += (size_t)d * b * 8;
  l.off_skf = o; o += d > 0 ? (size_t)T * b * 16 : 0;
  l.off_tri = o; o += has_tri ? (size_t)b * b * 8 : 0;
  l.off_dinv = o; o += has_tri ? (size_t)b * 8 : 0;
  l.off_ec = o; o += digits ? (size_t)NB * 32 : 0;
  l.bytes = o;
  return l;
}

// Tile height (64, 32 or 16) of the call's sketch schedule: the tallest for which a pass
// of a_max X columns and b_max panel columns keeps its digits of C in shared memory, 16 rows
// otherwise (a tile below 64 rows leaves warps without an update).
int rowpass_sketch_T(int a_max, int b_max, int d, int zeta) {
  for (int T = 64; T > 16; T /= 2) {
    const size_t need = tc_layout(a_max, b_max, T, 0, a_max > 0, true, false, false, d, sketch_sched_rec_bytes(T, d, zeta), a_max > 0).bytes;
    if (need <= 220 * 1024) return T;
  }
  return 16;
}

int rowpass_tc_launch(const RowPass& rpin, Arena* ar, cudaStream_t st, int* launches, int num_sms) {
  RowPass rp = rpin;
  const int d = rp.sk_d > 0 ? rp.sk_d : 0;
  // A tensor copy's coordinates are 32 bits wide.  Longer arrays come in without it in the sketch
  // passes, which no other kernel serves; the others go to rowpass_kernel.
  const bool long_rows = rp.n >= ((int64_t)1 << 31) - 1024;
  if (rp.sk_gd > 0 || (long_rows && d == 0)) return RBO_ERR_ARG;
  if (d > 0 && (rp.acc_x || rp.acc_y)) return RBO_ERR_ARG;  // a sketch pass has no Gram
  if (!rp.C && !rp.acc_x) rp.a = 0;  // X is not read
  const int a = rp.a, b = rp.b;
  const int ax = rp.acc_x ? a : 0;
  const int zr = ax + (rp.acc_y ? b : 0), no = zr * b, L = no + d * b;
  const bool hc = rp.C != nullptr;
  // Panels of more than 8 columns multiply by the inverse on the tensor cores where the
  // caller vouches for the factor (2^22 rows, b = 30, alone: 3717 us of substitution on the
  // float64 pipe, 1059 us); narrow ones substitute (2^22 x 61, b = 5, with the Gram: 674 us
  // against 897 by the inverse)
  bool want_inv = rp.Tri && rp.Inv && !hc && b > 8;
  // Gram items of a chunk: for every 8 columns of Y' (16 in wide kernels), the 16-column
  // groups of Z down to the block's diagonal
  const bool y_only = hc && !rp.Tri && ax == 0 && rp.acc_y && b > 8;
  int nblk = 0, q = 0, blk_start[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  auto count_items = [&]() {
    const int w = want_inv || y_only ? 16 : 8;
    nblk = (b + w - 1) / w;
    for (int k = 0; k < nblk; ++k) {
      const int need = zr == 0 ? 0 : ax + (rp.acc_y ? std::min(b, w * k + w) : 0);
      blk_start[k + 1] = blk_start[k] + (need + 15) / 16;
    }
    q = blk_start[nblk];
  };
  count_items();
  // Tile height and chunk.  Four items a tile keep the four warps busy in one turn, and long
  // chunks spare scans, conversions and joins of the sums (2^22 x 61, chunks of 32 -> 64 rows
  // at q = 3: 484 -> 470 us; more turns of shorter chunks, q = 1 in 64-row tiles: 494 us); a
  // chunk of 32 needs no conversion of its sums.  Solve + general Gram (XL: no second X stage)
  // takes the tallest tiles: 128-row chunks there, 674 -> 572 us (their sums stay below
  // 7 * 128 * 2^14 < 2^24).  Passes without a Gram take tiles of about 20 KB; sketch passes
  // those of the schedule.
  int T = 64, kc = 64;
  const bool narrow_gram = ax > 0 && b <= 8 && !rp.C;
  if (d > 0) {
    T = rp.sk.T;
  } else if (q == 0) {
    const int blk = tc_blk_bytes(a, rp.C ? 16 : 8) + tc_blk_bytes(b, 8);
    while (T < 256 && blk * (2 * T / 16) <= 20 * 1024) T *= 2;
  } else if (want_inv || y_only) {
    T = q == 1 ? 128 : 64;
    kc = q <= 2 ? 32 : 64;
  } else if (narrow_gram && rp.Tri) {
    T = q == 1 ? 256 : 128;
    kc = q <= 2 ? 64 : 128;
  } else if (q == 1) {
    // update + sym8: an X stage of at most 32 KB (2^22 x 61: 539 us against 566 with 64 rows for
    // every a and 581 with 128)
    const bool narrow = a + b <= 16, upd = rp.C && ax == 0;
    T = upd ? (a <= 16 ? 256 : (a <= 32 ? 128 : 64)) : (narrow ? 256 : 128);
    kc = narrow ? 64 : 32;
  } else if (q <= (narrow_gram ? 2 : 3)) {
    kc = 32;
  }
  // few rows: shorter tiles while they leave SMs without one
  while (d == 0 && T > 64 && (rp.n + T - 1) / T < 2 * (int64_t)num_sms) {
    T /= 2;
    kc = std::max(16, kc / 2);
  }
  auto kernel_of = [&](int tri) {
    if (y_only) return tc_kernel_g3();
    if (rp.elementwise && ax > 0 && !hc && !rp.Tri) return tc_kernel_g4();
    return q == 0 ? tc_kernel_g0(hc, tri, d > 0) : (ax == 0 && b <= 8 ? tc_kernel_g2(hc, tri) : tc_kernel_g1(hc, tri));
  };
  TcKernel kern = kernel_of(want_inv ? 2 : (rp.Tri ? 1 : 0));
  if (!kern) return RBO_ERR_ARG;
  int limit = tc_smem_limit((const void*)kern);
  const size_t epi_bytes = ((size_t)L + 2) * 8 + epilogue_doubles(rp) * 8;
  TcLayout l;
  size_t smem = 0;
  const bool gen = q > 0 && !(ax == 0 && b <= 8) && !y_only;  // general Gram
  const bool xs = rp.C ? !gen : (rp.Tri && gen);   // as the kernels' XS
  bool digits = rp.C != nullptr || want_inv;
  for (;;) {
    kc = (ax == 0 && b <= 8) ? std::max(16, T / 4) : std::min(kc, T);  // sym8: the warps' own rows
    l = tc_layout(a, b, T, q * (T / kc) * (want_inv || y_only ? 2 : 1), rp.C != nullptr, digits, rp.Tri != nullptr, want_inv && digits, d,
                  d > 0 ? rp.sk.rec_bytes : 0, xs);
    smem = std::max(l.bytes + 1024, epi_bytes);  // the tiles start at the next multiple of 1024
    if ((long long)smem <= limit) break;
    if (T > 16 && d == 0) T /= 2;
    else if (digits) {  // C stays float64, a factor is substituted
      digits = false;
      if (want_inv) {
        want_inv = false;
        count_items();
        kern = kernel_of(1);
        if (!kern) return RBO_ERR_ARG;
        limit = tc_smem_limit((const void*)kern);
      }
    } else return RBO_ERR_ARG;
  }
  const int ntiles = (int)((rp.n + T - 1) / T);
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, TC_NT, smem) != cudaSuccess) {
    cudaGetLastError();
    occ = 1;
  }
  int G = std::min(ntiles, std::min(std::max(occ, 1), 8) * num_sms);
  if (rp.max_ctas > 0) G = std::min(G, rp.max_ctas);
  if (G < 1) G = 1;
  const int ngroups = (G + GROUP - 1) / GROUP;

  TcDev D;
  PassDev& P = D.P;
  P = PassDev();
  P.p = rp;
  P.T = T;
  P.ntiles = ntiles;
  P.items = q * (T / kc);
  P.kc = kc;
  P.nblk = nblk;
  for (int k = 0; k < 9; ++k) P.blk_start[k] = blk_start[k];
  // (the leading dimension of a single column does not matter)
  const int64_t ldx = a == 1 ? rp.ldx + (rp.ldx & 1) : rp.ldx, ldy = b == 1 ? rp.ldy + (rp.ldy & 1) : rp.ldy;
  const bool alignedX = a == 0 || (((uintptr_t)rp.X & 15) == 0 && ldx % 2 == 0);
  const bool alignedY = ((uintptr_t)rp.Y & 15) == 0 && ldy % 2 == 0;
  P.use_bulk = (alignedX && alignedY && !long_rows) ? 1 : 0;
  if (P.use_bulk) {
    int e = make_tensor_map(&D.tmY, rp.Y, rp.n, b, ldy);
    if (e == RBO_OK && a > 0) e = make_tensor_map(&D.tmX, rp.X, rp.n, a, ldx);
    if (e != RBO_OK) return e;
  }
  P.zr = zr;
  P.no = no;
  P.L = L;
  P.ngroups = ngroups;
  P.status = ar->status;
  P.xblk = l.xblk;
  P.yblk = l.yblk;
  P.stage_bytes = (int)l.stage_bytes;
  P.off_c = (int)l.off_c;
  P.off_ec = (int)l.off_ec;
  P.off_acc = (int)l.off_acc;
  P.off_tri = (int)l.off_tri;
  P.off_dinv = (int)l.off_dinv;
  P.off_sk = (int)l.off_sk;
  P.off_skf = (int)l.off_skf;
  P.c_digits = rp.C && digits ? 1 : 0;
  P.off_red = 0;
  if (L > 0) {
    const size_t need = ((size_t)G * L + (size_t)ngroups * L) * 8;
    if (ar->red == nullptr || need > ar->red_bytes) return RBO_ERR_NOMEM;
    if (ngroups + 1 > ar->n_tickets) return RBO_ERR_NOMEM;
    P.partials = ar->red;
    P.gpart = ar->red + (size_t)G * L;
    P.tickets = ar->tickets;
    ar->gpart = P.gpart;
    ar->ngroups = ngroups;
  }
  ProfToken tok = prof_start(st);
  kern<<<G, TC_NT, smem, st>>>(D);
  if (prof_on()) {
    const double nn = (double)rp.n, A = a, B = b;
    const double by = 8.0 * nn * (A + B + (rp.write_y ? B : 0.0));
    double fl = 0.0;
    if (rp.C) fl += 2.0 * nn * A * B;
    if (rp.Tri) fl += nn * B * B;
    if (rp.acc_x) fl += 2.0 * nn * A * B;
    if (rp.acc_y) fl += nn * B * (B + 1.0);
    if (d > 0) fl += nn * (double)rp.sk_zeta * B;
    prof_stop(tok, st, 0, by, fl, rp.tag);
  }
  if (launches) ++*launches;
  return note_cuda(cudaGetLastError());
}

}  // namespace rbo
