// FP64 products on the tensor cores, by exact digits (an error-free splitting
// in the manner of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012,
// with fixed instead of floating point slices).
//
// On this GPU the FP64 pipe issues two multiply-adds per clock and SM, 1/64 of
// the FP32 rate, so FP64 matrix products (the GenEO band factorisations and
// their solves with eight right-hand sides) run on the f16 tensor pipe instead
// (mma.sync m16n8k16, measured at 600 TFLOP/s dense).  A number x with
// |x| < 2^G becomes the 63-bit integer X = x 2^(62-G), split into seven signed
// digits of radix 2^9,
//   X = sum_s d_s 2^(9 (6 - s)),  |d_s| <= 256,
// which FP16 holds exactly.  Products of digits are integers below 2^16, and
// over 32 terms and at most seven digit pairs their FP32 sums stay below 2^24,
// so every level sum S_l = sum_{s+t=l} sum_k d_s e_t is exact, in any order.
// Levels 0..6 are kept; what is dropped is below 2^-61 of the scales' product
// for a 32-term sum.  Two 64-bit integers, hi = levels 0..3 and lo = levels
// 4..6, carry sums over many tiles without rounding:
//   x . y = (hi 2^27 + lo) 2^(G_x + G_y - 70).
// A row of a Cholesky factor is bounded by the square root of its diagonal
// entry, |L_ik| <= sqrt(a_ii), so that is its scale, known before the
// factorisation: the error of a product is relative to sqrt(a_ii a_jj), as in
// the backward error bound of Cholesky itself, and smaller than FP64's by the
// guard bits.  Operands without such a bound of their own (a tile before its
// triangular solve, the inverse of a diagonal tile, right-hand sides) are
// scaled by those powers of two first, so that what shares a scale is of one
// natural size: multiplying the matrix by powers of four from row to row (and
// column to column) changes no digit.  Results are independent of the order of
// summation.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace geneo {

constexpr int kDig = 7;                          // digits per number
constexpr int kDigTile = kDig * 1024;            // halves of a 32 x 32 tile
constexpr uint32_t kDigBytes = kDigTile * 2;     // 14 KB
constexpr int kNoExp = -4000;                    // exponent of an all-zero scale group

// Smallest G with |v| < 2^G (kNoExp for zero and subnormal values).
__device__ __forceinline__ int exp_above(double v) {
  const int e = (__double2hiint(v) >> 20) & 0x7ff;
  return e ? e - 1022 : kNoExp;
}

// v 2^(62-G), rounded to an integer (|v| < 2^G).
__device__ __forceinline__ long long fixed62(double v, int G) {
  const long long b = __double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const int sh = e - 1013 - G;                   // 53-bit mantissa shifted by this
  if (e == 0 || sh < -54) return 0;
  long long m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
  m = sh >= 0 ? m << min(sh, 9) : (m + (1LL << (-sh - 1))) >> -sh;
  return b < 0 ? -m : m;
}

// Digit s of X, from X plus 256 in every digit but the first: bits in 0..512.
constexpr long long kDigBias = (1LL << 8) | (1LL << 17) | (1LL << 26) | (1LL << 35) | (1LL << 44) |
                               (1LL << 53);
__device__ __forceinline__ uint32_t digit_bits(long long xb, int s) {
  return s == 0 ? (uint32_t)((int)(xb >> 54) + 256) : (uint32_t)(xb >> (9 * (6 - s))) & 511u;
}
// 0x6400 | f is the half 1024 + f, exact for f < 1024; 0x6500 = 1280.
__device__ __forceinline__ __half digit_half(long long xb, int s) {
  return __hsub(__ushort_as_half((unsigned short)(0x6400u | digit_bits(xb, s))), __ushort_as_half(0x6500));
}

// Element (r, k) of a digit slice of a 32 x 32 tile: four 16 x 16 blocks, so
// that sixteen rows or sixteen columns of the tile are whole 512-byte pieces
// for a warp's copy, with rows of 32 bytes whose two 16-byte chunks change
// places every four rows: ldmatrix reads them without bank conflicts.
__device__ __forceinline__ int dig_index(int r, int k) {
  return (r >> 4) * 512 + (k >> 4) * 256 + (r & 15) * 16 + ((((k >> 3) ^ (r >> 2)) & 1) << 3) + (k & 7);
}

__device__ __forceinline__ uint32_t dig_smem(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm2(uint32_t (&r)[2], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
__device__ __forceinline__ void ldsm4_trans(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Byte offset in a digit slice of this lane's ldmatrix row: the A operand rows
// m0.. (16), columns k0.. (16); its transpose; and the B operand (rows n0.. (8)
// are columns of the product, k0.. (16); lanes 16.. repeat lanes 0..).
__device__ __forceinline__ uint32_t ldsm_a(int m0, int k0, int lane) {
  return 2 * dig_index(m0 + (lane & 15), k0 + 8 * (lane >> 4));
}
__device__ __forceinline__ uint32_t ldsm_at(int m0, int k0, int lane) {
  return 2 * dig_index(k0 + (lane & 7) + 8 * (lane >> 4), m0 + 8 * ((lane >> 3) & 1));
}
__device__ __forceinline__ uint32_t ldsm_b(int n0, int k0, int lane) {
  return 2 * dig_index(n0 + (lane & 7), k0 + 8 * ((lane >> 3) & 1));
}

// The two integer parts of one product entry from its level sums.  Levels below
// M, whose sums stay within 2^22 (over 16 terms the first four, over 32 the first
// two), start at 1.5 2^23 (level_start) and are read from the bits: conversions
// issue at an eighth of the rate of integer instructions.
constexpr float kLevelOne = 12582912.f;          // 1.5 2^23: unit spacing, 2^22 either way
template <int M>
__device__ __forceinline__ void level_start(float (&S)[kDig][4]) {
#pragma unroll
  for (int l = 0; l < kDig; ++l)
#pragma unroll
    for (int e = 0; e < 4; ++e) S[l][e] = l < M ? kLevelOne : 0.f;
}
template <int M = 0>
__device__ __forceinline__ void level_parts(const float (&S)[kDig][4], int e, long long &hi,
                                            long long &lo) {
  int s[kDig];
#pragma unroll
  for (int l = 0; l < kDig; ++l)
    s[l] = l < M ? __float_as_int(S[l][e]) - 0x4b400000 : __float2int_rn(S[l][e]);
  hi = (long long)(s[0] * 512 + s[1]) * 262144 + ((long long)s[2] * 512 + s[3]);
  lo = (long long)s[4] * 262144 + ((long long)s[5] * 512 + s[6]);
}

// (hi 2^27 + lo) 2^(e - 70), zero below the normal range: the integer as a double,
// whose exponent field is then moved (a factor 2^(e - 70) may itself leave the range).
__device__ __forceinline__ double parts_value(long long hi, long long lo, int e) {
  const double v = fma((double)hi, 134217728.0, (double)lo);
  const int h = __double2hiint(v), bv = (h >> 20) & 0x7ff, be = bv + e - 70;
  if (bv == 0 || be < 1) return 0.0;
  if (be > 2046) return __hiloint2double((h & 0x80000000) | 0x7ff00000, 0);
  return __hiloint2double(h + ((e - 70) << 20), __double2loint(v));
}

// m 2^(ex - 64) with 2^63 <= m < 2^64, or zero (m = 0, ex <= kNoExp), and a sign.
struct Fixed {
  unsigned long long m;
  int ex;
  bool neg;
  // The number times 2^(62 - G), rounded to an integer (ex <= G).
  __device__ __forceinline__ long long at(int G) const {
    const int sh = 2 + G - ex;
    const long long x = m == 0 || sh > 64 ? 0 : (long long)((m >> (sh - 1)) + 1) >> 1;
    return neg ? -x : x;
  }
  // As a double, rounded to nearest; zero below the normal range.
  __device__ __forceinline__ double value() const {
    const int be = ex + 1022;
    if (m == 0 || be < 1) return 0.0;
    const unsigned long long b = be > 2046 ? 0x7ff0000000000000ULL
                                           : ((unsigned long long)(be - 1) << 52) + (m >> 11) + ((m >> 10) & 1);
    return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ULL : 0)));
  }
};

// (hi 2^27 + lo) 2^(f - 70), to 64 bits.
__device__ __forceinline__ Fixed fixed_of(long long hi, long long lo, int f) {
  unsigned long long l = ((unsigned long long)hi << 27) + (unsigned long long)lo;
  unsigned long long h = (unsigned long long)((hi >> 37) + (lo >> 63)) + (l < (unsigned long long)lo);
  const bool neg = (long long)h < 0;
  if (neg) {
    l = 0 - l;
    h = ~h + (l == 0);
  }
  const bool wide = h != 0;
  const unsigned long long t = wide ? h : l;
  const int z = __clzll(t);                      // 64 if zero
  unsigned long long m = t << (z & 63);
  if (wide && z) m |= l >> (64 - z);
  return t ? Fixed{m, (wide ? 58 : -6) - z + f, neg} : Fixed{0, kNoExp, false};
}

// The integer M with v = M 2^(exp_above(v) - 53), |M| < 2^53 (zero for subnormal v).
__device__ __forceinline__ long long mantissa53(double v) {
  const long long b = __double_as_longlong(v);
  if (!((b >> 52) & 0x7ff)) return 0;
  const long long m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
  return b < 0 ? -m : m;
}

// 16-byte asynchronous copies into shared memory, in groups of the issuing thread.
__device__ __forceinline__ void cp16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

}  // namespace geneo
