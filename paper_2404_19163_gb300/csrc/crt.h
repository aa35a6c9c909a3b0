// Modular (Chinese remainder) arithmetic of the residue products in k_ozmod.cu, shared by the
// host planner and the device kernels.  Plain C++ outside nvcc, so the arithmetic can be
// checked on the host.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define ZF_HD __host__ __device__
#else
#define ZF_HD
#endif

namespace zf {

constexpr int kCrtMax = 16;        // moduli of this table (crt_wide.h adds eight)
constexpr int kCrtMaxResidue = 128;  // largest |residue|: K-chunks of 2^24 / 128^2 = 1024 terms stay exact
constexpr int kCrtSubKb = (1 << 24) / (kCrtMaxResidue * kCrtMaxResidue) / 64;  // 64-wide K-blocks per chunk

// Pairwise coprime moduli up to 256, largest first: 2^8, then products of small primes and primes,
// so that the first k carry about 7.9 bits each and all sixteen multiply to about 2^125.38.  Residues
// |r| <= 128 are exact in BF16 (8 significand bits).
ZF_HD constexpr int crt_modulus(int i) {
  switch (i) {
    case 0: return 256;
    case 1: return 255;  // 3 5 17
    case 2: return 253;  // 11 23
    case 3: return 251;
    case 4: return 247;  // 13 19
    case 5: return 241;
    case 6: return 239;
    case 7: return 233;
    case 8: return 229;
    case 9: return 227;
    case 10: return 223;
    case 11: return 217;  // 7 31
    case 12: return 211;
    case 13: return 199;
    case 14: return 197;
    case 15: return 193;
    default: return 1;
  }
}

ZF_HD inline float crt_bits_f(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  memcpy(&f, &u, 4);
  return f;
#endif
}
ZF_HD inline unsigned crt_f_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  unsigned u;
  memcpy(&u, &f, 4);
  return u;
#endif
}

// Nearest integer (ties to even) of |x| < 2^22 with two FP32 additions: adding 1.5 * 2^23 leaves
// no fraction bits.
ZF_HD inline float crt_rint(float x) {
  const float C = 12582912.0f;
  return (x + C) - C;
}

ZF_HD inline double crt_bits_d(unsigned long long u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double d;
  memcpy(&d, &u, 8);
  return d;
#endif
}
ZF_HD inline int crt_clz64(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// (neg ? -x : x) 2^sc for the 128-bit magnitude x = hi 2^64 + lo, rounded once to the nearest double
// (ties to even), with integer operations only: GB300's FP64 pipe runs at a small fraction of its
// integer rate, and a reconstruction converts every entry.  Results outside the normal range go
// through ldexp of the exactly representable rounded significand.
ZF_HD inline double crt_to_double(unsigned long long hi, unsigned long long lo, bool neg, int sc) {
  if ((hi | lo) == 0ull) return 0.0;
  const int lz = hi ? crt_clz64(hi) : 64 + crt_clz64(lo);
  unsigned long long t, r;  // the magnitude shifted so that its leading one is bit 63 of t; r the rest
  if (lz >= 64) {
    t = lo << (lz - 64);
    r = 0ull;
  } else if (lz == 0) {
    t = hi;
    r = lo;
  } else {
    t = (hi << lz) | (lo >> (64 - lz));
    r = lo << lz;
  }
  unsigned long long m = t >> 11;  // 53 significant bits
  const bool round_bit = ((t >> 10) & 1ull) != 0ull, sticky = ((t & 0x3FFull) | r) != 0ull;
  if (round_bit && (sticky || (m & 1ull))) ++m;
  int e = 127 - lz + sc;  // value = m 2^(e - 52)
  if (m >> 53) {
    m >>= 1;
    ++e;
  }
  const int be = e + 1023;
  if (be <= 0 || be >= 2047) {
    const double v = ldexp((double)m, e - 52);
    return neg ? -v : v;
  }
  return crt_bits_d(((unsigned long long)neg << 63) | ((unsigned long long)be << 52) | (m & ((1ull << 52) - 1ull)));
}

// 2^e mod m in symmetric form (|c| <= m/2).
ZF_HD constexpr int crt_pow2_sym(int m, int e) {
  int r = 1 % m;
  for (int i = 0; i < e; ++i) r = (2 * r) % m;
  return 2 * r > m ? r - m : r;
}

// Residue modulo m of F = sum_k a_k 2^(14k) from its NP signed 14-bit parts (NP = 6 holds 84 bits), as the kernels take it
// (there on pairs of elements, one instruction for two).  x = sum_k a_k (2^(14k) mod m) with the symmetric |2^(14k) mod m|
// <= m/2 is an integer below 2^24 (exact), |x / m| <= 6 2^13.  The quotient's product and rounding are one operation: it errs
// by at most 6 2^13 2^-24 < 0.003 (1/m's rounding) before it is rounded, and |r| <= m 0.503 < 129 for m <= 255:
// |r| <= 128 (m = 256: exact quotient).
template <int NP>
ZF_HD inline float crt_residue_step(const float* a, int m) {
  const float fm = (float)m, inv = 1.0f / fm;
  float x = a[0];
  for (int k = 1; k < NP; ++k) x = fmaf(a[k], (float)crt_pow2_sym(m, 14 * k), x);
  return fmaf(-fm, fmaf(x, inv, 12582912.0f) - 12582912.0f, x);
}
// The signed 14-bit part v (below 2^14) of a value: the bits of 2^23 + v, minus 2^23, with the value's sign bit.
ZF_HD inline float crt_part_f(unsigned v, unsigned sign_bit) {
  return crt_bits_f(crt_f_bits(crt_bits_f(0x4B000000u | v) - 8388608.0f) ^ sign_bit);
}

// A residue product's sum to its CRT digit, as the product's epilogue takes it (there on pairs of columns, one
// instruction for two).  crt_step: x mod m for |x| <= 2^24 with the quotient's product and rounding in one operation; the
// quotient is off by at most |x / m| 2^-24 (inv's rounding), so |r| <= m (1/2 + 2^24 / 151 2^-24) < m 0.507.
// Two columns' sums of such residues share a float, r0 + 4096 r1, which is an exact integer that crt_unpack2 takes apart
// while |r0|, |r1| < 2048.  |r| <= m/2 + 1 and so <= 128; a fold reduces both sums to such residues again, and kCrtFoldSub
// steps from there stay within 15 * 128 = 1920.  crt_digit_sum: the digit s w mod m in [0, m) of a sum |s| < 2048, by
// floor(x / m) = rint((x + 1/2) / m - 1/2): the argument stays 1 / 2m >= 0.0019 from a tie and is computed
// to 0.0004.
constexpr int kCrtFoldSub = 14;
ZF_HD inline float crt_step(float x, float m, float inv) {
  return fmaf(-m, fmaf(x, inv, 12582912.0f) - 12582912.0f, x);
}
ZF_HD inline void crt_unpack2(float p, float* r0, float* r1) {
  *r1 = fmaf(p, 1.0f / 4096.0f, 12582912.0f) - 12582912.0f;
  *r0 = fmaf(-4096.0f, *r1, p);
}
ZF_HD inline float crt_digit_sum(float s, float m, float inv, float w) {
  const float x = s * w;
  return fmaf(-m, crt_rint(fmaf(x, inv, 0.5f * inv - 0.5f)), x);
}

}  // namespace zf
