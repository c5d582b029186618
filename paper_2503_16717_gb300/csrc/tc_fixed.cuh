// Float64 products on the fp16 tensor cores, from exact fixed-point digits.
//
// The float64 pipe of this GPU does 2 FMAs per SM and cycle, the fp16 tensor cores 1024
// through mma.sync (both measured), so the contractions of a row pass (X^T Y', y - x C)
// are formed from integers (Ozaki, Ogita, Oishi and Rump 2012):
//   - a group of values that share a scale (one column over a chunk of rows, or one row
//     over the columns) with largest exponent field E becomes x = +-F 2^(E - 1077), F the
//     55-bit integer (4 M) >> (E - e), M the 53-bit significand: values within a factor of
//     4 of the group's largest keep all their bits, any value is off by less than a quarter
//     of an ulp of the largest;
//   - F = sum_j d_j 2^(8 j), j = 0..6, with balanced digits -128 <= d_j <= 127 below the
//     top one, 0 <= d_6 <= 128: adding 128 to the six lower byte positions makes the bytes
//     d_j + 128 and d_6; a byte permute with 0x64 in the high half gives the fp16 value
//     1024 + byte of two elements, and one fused multiply-add by the signs turns it into
//     +-d_j, exact in fp16;
//   - digit products are at most 2^14 and are summed per level I + J (I, J = 6 - j) in the
//     float32 accumulators of mma.sync.m16n8k16: up to 128 terms of at most 7 pairs per
//     level stay below 2^24, so every sum is exact in any order;
//   - the levels 0..6 (28 digit pairs) are joined in 64-bit integers and enter the
//     float64 result with one conversion and one FMA.  The pairs left out (I + J >= 7)
//     weigh at most 6 * 2^54 / 2^108 < 2^-51.4 of the largest product of the group per
//     term (whose factors are at least 2^54 each), about 2^-55 root mean square over the
//     digits' signs; joining rounds at 2^-55 of it once per chunk.
// A group with a non-finite value, or with its largest value outside 2^+-463, is
// computed by float64 FMAs instead.  So is, where the Gram itself is asked for, an entry's chunk
// in which the large values of the two columns do not meet (tc_tile.cuh): there the error, which
// goes by the largest values, could exceed that of float64 sums, which goes by the products.
//
// Why the digits go from registers into mma.sync: every thread forms the digits of the
// fragment elements it owns, so no operand passes through shared or tensor memory
// between the conversion and the product, and no barrier separates them.  The conversion
// (about 11 half-rate integer operations per value) is the cost; the tensor cores are
// not the limit at 1024 MACs per SM and cycle.
#pragma once

#include <cuda_fp16.h>

#include "device_common.cuh"

namespace rbo {

constexpr int FX_EMIN = 560;    // smallest and largest exponent field of a group in
constexpr int FX_EMAX = 1486;   // fixed point (2^-463 .. 2^463)
constexpr int FX_EZERO = 559;   // scale of a group of zeros
constexpr uint32_t FX_MAGIC = 0x4B400000u;  // 1.5 * 2^23: float bits minus this = integer

// twice the largest |x| high word and the OR of low words of the scanned values
struct FxMax {
  uint32_t m = 0u, nz = 0u;
  __device__ __forceinline__ void add(double a, double b) {
    const uint32_t u = (uint32_t)__double2hiint(a), v = (uint32_t)__double2hiint(b);
    m = max(m, max(u + u, v + v));
    nz |= (uint32_t)__double2loint(a) | (uint32_t)__double2loint(b);
  }
  // over the 4 lanes that share a group (lane & 3)
  __device__ __forceinline__ void reduce4() {
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    nz |= __shfl_xor_sync(0xffffffffu, nz, 1);
    nz |= __shfl_xor_sync(0xffffffffu, nz, 2);
  }
  // exponent field to scale by; 0 when the group needs the float64 path (a subnormal
  // group with nonzero bits counts as below FX_EMIN)
  __device__ __forceinline__ int scale() const {
    const int e = (int)(m >> 21);
    if ((m | nz) == 0u) return FX_EZERO;
    return (e >= FX_EMIN && e <= FX_EMAX) ? e : 0;
  }
};

// Scale of a group with exponent field E: key - 2 h (h the high word of a value) has
// E - e in its top 11 bits, and the high word of 4 M is (h : l) << 2 with the exponent
// bits replaced by the leading one, (h : l << 2)_hi + lead + ((E - e) << 22) modulo 2^32
struct FxScale {
  uint32_t key, lead;
};
__device__ __forceinline__ FxScale fx_scale(int E) {
  return FxScale{((uint32_t)E << 21) | 0x1FFFFFu, (1u - (uint32_t)E) << 22};
}

// A value as an integer of at most 2^54 on the scale of exponent field E (unit
// 2^(E - 1076)), rounded to nearest, ties away from zero; zero and subnormal values give 0
// (values past the scale give garbage)
__device__ __forceinline__ long long fx_round54(double v, int E) {
  const uint32_t l = (uint32_t)__double2loint(v), h = (uint32_t)__double2hiint(v);
  const uint32_t e = (h >> 20) & 0x7FFu;
  const uint32_t m = (__funnelshift_l(l, h, 2) & 0x3FFFFFu) | 0x400000u;  // high word of 4 M
  uint64_t F;
  asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tshr.u64 t, t, %3;\n\tadd.u64 t, t, 1;\n\tshr.u64 %0, t, 1;\n\t}"
      : "=l"(F)
      : "r"(l << 2), "r"(m), "r"(e == 0u ? 64u : (uint32_t)E - e));
  return (h >> 31) ? -(long long)F : (long long)F;
}

// Masks of the digit extraction.  They are made opaque to the compiler so that they stay
// in registers: a three-input logic operation takes one immediate only, and with two it
// becomes two operations.
struct FxMask {
  uint32_t sign, one, m3, k3, k64;
};
__device__ __forceinline__ FxMask fx_masks() {
  FxMask k;
  asm volatile("mov.b32 %0, 0x80008000;" : "=r"(k.sign));
  asm volatile("mov.b32 %0, 0x3C003C00;" : "=r"(k.one));
  asm volatile("mov.b32 %0, 0x00FF00FF;" : "=r"(k.m3));
  asm volatile("mov.b32 %0, 0x64006400;" : "=r"(k.k3));
  asm volatile("mov.b32 %0, 0x64646464;" : "=r"(k.k64));
  return k;
}
__device__ __forceinline__ uint32_t fx_and_or(uint32_t x, uint32_t m, uint32_t o) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(x), "r"(m), "r"(o));  // (x & m) | o
  return r;
}

// Two values of one digit pair: biased 55-bit integers and the signs as fp16 factors
struct FxPair {
  uint32_t lo0, hi0, lo1, hi1;
  __half2 s, c;   // +-1, -+1152
};

__device__ __forceinline__ void fx_fix(double v, FxScale sc, uint32_t& lo, uint32_t& hi) {
  const uint32_t l = (uint32_t)__double2loint(v), h = (uint32_t)__double2hiint(v);
  const uint32_t sh = (sc.key - (h + h)) >> 21;                                  // E - e
  const uint32_t m = __funnelshift_l(l, h, 2) + sc.lead + (sh << 22);            // high word of 4 M
  uint64_t F;
  asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tshr.u64 t, t, %3;\n\tadd.u64 %0, t, 0x6400808080808080;\n\t}"
      : "=l"(F)
      : "r"(l << 2), "r"(m), "r"(sh));
  lo = (uint32_t)F;
  hi = (uint32_t)(F >> 32);
}

__device__ __forceinline__ FxPair fx_pair(double v0, double v1, FxScale sc, const FxMask& k) {
  FxPair p;
  fx_fix(v0, sc, p.lo0, p.hi0);
  fx_fix(v1, sc, p.lo1, p.hi1);
  const uint32_t sg = __byte_perm((uint32_t)__double2hiint(v0), (uint32_t)__double2hiint(v1), 0x7030);
  const uint32_t s = fx_and_or(sg, k.sign, k.one);
  p.s = *reinterpret_cast<const __half2*>(&s);
  p.c = __hmul2(p.s, __half2half2(__ushort_as_half(0xE480)));
  return p;
}

// Digit I (0 = most significant) of the pair as fp16x2.  Digit 3 (the top byte of the low
// words) must be taken before fx_mask_low, digits 4..6 after it.
template <int I>
__device__ __forceinline__ uint32_t fx_digit(const FxPair& p, const FxMask& k) {
  uint32_t x;
  if (I == 0) x = __byte_perm(p.hi0, p.hi1, 0x7632);
  else if (I == 1) x = __byte_perm(p.hi0, p.hi1, 0x7531);
  else if (I == 2) x = __byte_perm(p.hi0, p.hi1, 0x7430);
  else if (I == 3) x = fx_and_or(__byte_perm(p.lo0, p.lo1, 0x0703), k.m3, k.k3);
  else if (I == 4) x = __byte_perm(p.lo0, p.lo1, 0x7632);
  else if (I == 5) x = __byte_perm(p.lo0, p.lo1, 0x7531);
  else x = __byte_perm(p.lo0, p.lo1, 0x7430);
  // the top byte carries no offset: -+1024 instead of -+1152
  const __half2 c = I == 0 ? __hfma2(p.s, __half2half2(__ushort_as_half(0x5800)), p.c) : p.c;
  const __half2 d = __hfma2(*reinterpret_cast<const __half2*>(&x), p.s, c);
  return *reinterpret_cast<const uint32_t*>(&d);
}
__device__ __forceinline__ void fx_mask_low(FxPair& p, const FxMask& k) {
  p.lo0 = __byte_perm(p.lo0, k.k64, 0x4210);
  p.lo1 = __byte_perm(p.lo1, k.k64, 0x4210);
}

__device__ __forceinline__ void fx_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                       uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// the same with another addend: d = A B + c
__device__ __forceinline__ void fx_mma_first(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                             uint32_t b0, uint32_t b1, const float (&c)[4]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %11, %12, %13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// All pairs I + J <= 6 of one K step: A = four pairs of values, p[row half][K half] (rows
// g / g + 8), B = digits bd[J][K half]
// FIRST: the first step of a sum, which starts from `init` instead of the accumulators.
// NT column tiles of B share the digits of A, which are two thirds of a step's instructions.
// sizes: unless null, the same sums of the sizes of the top digits alone.
template <int I, bool FIRST, int NT>
__device__ __forceinline__ void fx_level(float (&acc)[NT][7][4], const FxPair& p00, const FxPair& p10,
                                         const FxPair& p01, const FxPair& p11, const uint32_t (&bd)[NT][7][2],
                                         const FxMask& k, const float (&init)[4], float (*sizes)[4]) {
  const uint32_t a0 = fx_digit<I>(p00, k), a1 = fx_digit<I>(p10, k), a2 = fx_digit<I>(p01, k),
                 a3 = fx_digit<I>(p11, k);
#pragma unroll
  for (int h = 0; h < NT; ++h)
#pragma unroll
    for (int J = 0; J + I <= 6; ++J) {
      if (FIRST && I == 0) fx_mma_first(acc[h][J], a0, a1, a2, a3, bd[h][J][0], bd[h][J][1], init);
      else fx_mma(acc[h][I + J], a0, a1, a2, a3, bd[h][J][0], bd[h][J][1]);
    }
  if (I == 0 && sizes != nullptr) {
    const float zero[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int h = 0; h < NT; ++h) {
      const uint32_t b0 = bd[h][0][0] & ~k.sign, b1 = bd[h][0][1] & ~k.sign;
      if (FIRST) fx_mma_first(sizes[h], a0 & ~k.sign, a1 & ~k.sign, a2 & ~k.sign, a3 & ~k.sign, b0, b1, zero);
      else fx_mma(sizes[h], a0 & ~k.sign, a1 & ~k.sign, a2 & ~k.sign, a3 & ~k.sign, b0, b1);
    }
  }
}
template <bool FIRST, int NT>
__device__ __forceinline__ void fx_step(float (&acc)[NT][7][4], FxPair& p00, FxPair& p10, FxPair& p01,
                                        FxPair& p11, const uint32_t (&bd)[NT][7][2], const FxMask& k,
                                        const float (&init)[4], float (*sizes)[4] = nullptr) {
  fx_level<0, FIRST, NT>(acc, p00, p10, p01, p11, bd, k, init, sizes);
  fx_level<1, FIRST, NT>(acc, p00, p10, p01, p11, bd, k, init, nullptr);
  fx_level<2, FIRST, NT>(acc, p00, p10, p01, p11, bd, k, init, nullptr);
  fx_level<3, FIRST, NT>(acc, p00, p10, p01, p11, bd, k, init, nullptr);
  fx_mask_low(p00, k);
  fx_mask_low(p10, k);
  fx_mask_low(p01, k);
  fx_mask_low(p11, k);
  fx_level<4, FIRST, NT>(acc, p00, p10, p01, p11, bd, k, init, nullptr);
  fx_level<5, FIRST, NT>(acc, p00, p10, p01, p11, bd, k, init, nullptr);
  fx_level<6, FIRST, NT>(acc, p00, p10, p01, p11, bd, k, init, nullptr);
}
// digits of a B fragment (K pairs q0: 2t, 2t+1 and q1: 2t+8, 2t+9 of column g)
__device__ __forceinline__ void fx_bdigits(FxPair& q0, FxPair& q1, uint32_t (&bd)[7][2], const FxMask& k) {
  bd[0][0] = fx_digit<0>(q0, k); bd[0][1] = fx_digit<0>(q1, k);
  bd[1][0] = fx_digit<1>(q0, k); bd[1][1] = fx_digit<1>(q1, k);
  bd[2][0] = fx_digit<2>(q0, k); bd[2][1] = fx_digit<2>(q1, k);
  bd[3][0] = fx_digit<3>(q0, k); bd[3][1] = fx_digit<3>(q1, k);
  fx_mask_low(q0, k);
  fx_mask_low(q1, k);
  bd[4][0] = fx_digit<4>(q0, k); bd[4][1] = fx_digit<4>(q1, k);
  bd[5][0] = fx_digit<5>(q0, k); bd[5][1] = fx_digit<5>(q1, k);
  bd[6][0] = fx_digit<6>(q0, k); bd[6][1] = fx_digit<6>(q1, k);
}

// Accumulators start at 1.5 * 2^23 while the sums stay below 2^22 (at most 32 terms), so
// that the integer is the bit difference; otherwise at 0, converted.
__device__ __forceinline__ void fx_init(float (&c)[4], bool small) {
  const float v = small ? __uint_as_float(FX_MAGIC) : 0.0f;
#pragma unroll
  for (int o = 0; o < 4; ++o) c[o] = v;
}
// the sums as integers, in place
__device__ __forceinline__ void fx_ints(float (&acc)[7][4], bool small) {
  if (small) {
#pragma unroll
    for (int l = 0; l < 7; ++l)
#pragma unroll
      for (int o = 0; o < 4; ++o) acc[l][o] = __int_as_float(__float_as_int(acc[l][o]) - (int)FX_MAGIC);
  } else {
#pragma unroll
    for (int l = 0; l < 7; ++l)
#pragma unroll
      for (int o = 0; o < 4; ++o) acc[l][o] = __int_as_float(__float2int_rn(acc[l][o]));
  }
}
// Output o of the level sums (after fx_ints): sum_l S_l 2^(8 (12 - l)) in units of 2^55, the
// levels joined in integers (128 terms: |S_l| <= (l + 1) 2^21, so that the joined value is
// below 2^62.1)
__device__ __forceinline__ double fx_join(const float (&acc)[7][4], int o) {
  int s[7];
#pragma unroll
  for (int l = 0; l < 7; ++l) s[l] = __float_as_int(acc[l][o]);
  long long t1, t2;
  asm("{\n\t.reg .b64 v;\n\tcvt.s64.s32 v, %2;\n\tmad.wide.s32 %0, %1, 65536, v;\n\t}"
      : "=l"(t1)
      : "r"(s[0] * 256 + s[1]), "r"(s[2] * 256 + s[3]));
  asm("{\n\t.reg .b64 v;\n\tcvt.s64.s32 v, %3;\n\tmad.wide.s32 v, %2, 256, v;\n\tmad.wide.s32 %0, %1, 65536, v;\n\t}"
      : "=l"(t2)
      : "r"(s[4]), "r"(s[5]), "r"(s[6] + 64));
  return (double)((t1 << 17) + (t2 >> 7));
}
// 2^(Ex + Ey - 2099): weight of fx_join for scales Ex, Ey
__device__ __forceinline__ double fx_weight(int Ex, int Ey) {
  return __hiloint2double((Ex + Ey - 1076) << 20, 0);
}

}  // namespace rbo
