// Reference forms of the CRT arithmetic for the host checks: limb sums over the digits, scalar residues and digits.  They are
// independent of the kernels' forms (crt_residue_step, crt_step, crt_digit_sum, crt_combine_value), which the checks hold
// against them or against integers; no kernel and no host code of the library uses them.  Included by crt_wide.h outside nvcc.
#pragma once
#include "crt_wide.h"

namespace zf {

// The integer nearest (ties to even) to |x| < 2^22 with FP32 and integer operations only.
ZF_HD inline int crt_rint_i(float x) { return (int)(crt_f_bits(x + 12582912.0f) - 0x4B400000u); }
// An integer 0 <= y < 2^23 as a float, exactly (the bits of 2^23 + y, minus 2^23).
ZF_HD inline float crt_u2f(unsigned y) { return crt_bits_f(0x4B000000u | y) - 8388608.0f; }

// The five 14-bit parts of a fixed-point value F (|F| <= 2^62), signed, as floats:
// F = sum_k a_k 2^(14k), |a_k| < 2^14.
ZF_HD inline void crt_parts(long long F, float (&a)[5]) {
  const unsigned long long u = F < 0 ? 0ull - (unsigned long long)F : (unsigned long long)F;
  const float sg = F < 0 ? -1.0f : 1.0f;
  // a 14-bit integer v as a float: the bits of 2^23 + v, minus 2^23
  for (int k = 0; k < 5; ++k)
    a[k] = sg * (crt_bits_f(0x4B000000u | (unsigned)((u >> (14 * k)) & 0x3FFFu)) - 8388608.0f);
}

// Residue of F modulo m from its first NP parts (NP = 4 when |F| < 2^56), in FP32: x = sum_k a_k
// (2^(14k) mod m), with |a_k| < 2^14 and the symmetric |2^(14k) mod m| <= m/2, is an integer with
// |x / m| < 5 2^13, below 2^24 (exact).  r = x - m rint(x / m) is congruent to F; the FP32 quotient
// (1/m and the product each rounded once) errs by at most |x / m| 2^-23 < 0.0049, so rint is at most one
// step from the nearest integer and |r| <= m (1/2 + 0.0049) < 128.8 for m <= 255, |r| <= 128; for
// m = 256 the quotient is exact and |r| <= 128 too.  (Not always the symmetric residue, but within the
// bound the residue products need.)
template <int NP = 5>
ZF_HD inline float crt_residue_f(const float (&a)[5], int m) {
  const float fm = (float)m;
  float x = fmaf(a[3], (float)crt_pow2_sym(m, 42),
                 fmaf(a[2], (float)crt_pow2_sym(m, 28), fmaf(a[1], (float)crt_pow2_sym(m, 14), a[0])));
  if (NP > 4) x = fmaf(a[4], (float)crt_pow2_sym(m, 56), x);
  return fmaf(-fm, crt_rint(x * (1.0f / fm)), x);
}

// x mod m for an integer-valued float |x| <= 2^24 and m >= 13, inv = FP32(1 / m): congruent, and
// within 0.66 m of 0.  The FP32 quotient x * inv carries a relative error of at most 2^-23 (inv and
// the product each rounded once), so it is off by at most 2^24 / 13 * 2^-23 = 0.154 from x / m (well
// inside crt_rint's range); rint is then at most one step from the nearest integer, |x - m rint| <=
// m (1/2 + 0.154), and the fma is exact because that difference is an integer below 2^24.
ZF_HD inline float crt_fmod_sym(float x, float m, float inv) { return fmaf(-m, crt_rint(x * inv), x); }

// The CRT digit of an exact residue-product sum v (integer-valued float, |v| <= 2^24): y = (v mod m) w
// mod m in [0, m), w = (M / m)^-1 mod m the plan's weight of this modulus.  |v mod m| <= 0.66 m <= 169
// and w < 256, so the product stays an exact integer below 2^16, and its second reduction leaves
// |y| <= 0.66 m, which the shift of negative values by m takes into [0, m).
ZF_HD inline float crt_digit(float v, float m, float inv, float w) {
  float y = crt_fmod_sym(crt_fmod_sym(v, m, inv) * w, m, inv);
  return y < 0.0f ? y + m : y;
}

// Reconstruction constants of the first nmod moduli: M = prod m_i, P_i = M / m_i as four
// 32-bit limbs, w_i = P_i^-1 mod m_i.
struct CrtPlan {
  int nmod;
  int m[kCrtMax];
  int w[kCrtMax];
  float inv[kCrtMax];
  float fm[kCrtMax], fw[kCrtMax];  // m and w as floats
  unsigned P[kCrtMax][4];
  unsigned M[4];
};

// Accumulates sum_i y_i P_i (y_i congruent to (C mod m_i) w_i modulo m_i, y_i < 2^10) per 32-bit limb
// without carries (each limb sum stays below 2^46) and sum_i y_i / m_i in FP32.  That sum equals q + C / M for
// an integer q; with |C| < M / 4 and an FP32 error far below 1/4, q = round(sum) and
// C = sum_i y_i P_i - q M, formed modulo 2^128 (exact, since |C| < 2^125).
struct CrtAcc {
  unsigned long long L[4];
  float S;
  ZF_HD void clear() {
    L[0] = L[1] = L[2] = L[3] = 0ull;
    S = 0.0f;
  }
  // Adds a sum y of CRT digits of modulus t (one per digit plane, each in [0, m_t), so y < 2^10).  The
  // digits need no reduction: any y congruent to (C mod m_t) w_t gives sum_t y_t P_t = C (mod M), and
  // sum_t y_t / m_t is still q + C / M for an integer q (below 2^7 here, far from FP32's limits).
  ZF_HD void add_y(const CrtPlan& p, int t, unsigned y) {
    S = fmaf(crt_u2f(y), p.inv[t], S);
    for (int l = 0; l < 4; ++l) L[l] += (unsigned long long)y * p.P[t][l];
  }
  // C 2^sc in FP64, rounded once (crt_to_double).
  ZF_HD double value(const CrtPlan& p, int sc) const {
    const long long q = crt_rint_i(S);
    long long t0 = (long long)L[0] - q * (long long)p.M[0];
    long long t1 = (long long)L[1] - q * (long long)p.M[1] + (t0 >> 32);
    long long t2 = (long long)L[2] - q * (long long)p.M[2] + (t1 >> 32);
    long long t3 = (long long)L[3] - q * (long long)p.M[3] + (t2 >> 32);
    const unsigned l0 = (unsigned)t0, l1 = (unsigned)t1, l2 = (unsigned)t2, l3 = (unsigned)t3;
    unsigned long long hi = ((unsigned long long)l3 << 32) | l2, lo = ((unsigned long long)l1 << 32) | l0;
    const bool neg = (l3 >> 31) != 0u;
    if (neg) {
      lo = ~lo + 1ull;
      hi = ~hi + (lo == 0ull ? 1ull : 0ull);
    }
    return crt_to_double(hi, lo, neg, sc);
  }
};

// The moduli count that makes M = m_0 ... m_{k-1} exceed 2^bits (0 if all sixteen do not), with
// the reconstruction constants.
inline int crt_plan(double bits, CrtPlan* p) {
  unsigned __int128 M = 1;
  int k = 0;
  double lb = 0.0;
  while (k < kCrtMax && lb <= bits) {
    M *= (unsigned)crt_modulus(k);
    lb += log2((double)crt_modulus(k));
    ++k;
  }
  if (lb <= bits) return 0;
  p->nmod = k;
  for (int i = 0; i < kCrtMax; ++i) {
    const unsigned m = i < k ? (unsigned)crt_modulus(i) : 1u;
    p->m[i] = (int)m;
    p->inv[i] = 1.0f / (float)m;
    p->fm[i] = (float)m;
    p->w[i] = 0;
    p->fw[i] = 0.0f;
    for (int l = 0; l < 4; ++l) p->P[i][l] = 0u;
    if (i >= k) continue;
    const unsigned __int128 P = M / m;
    for (int l = 0; l < 4; ++l) p->P[i][l] = (unsigned)(P >> (32 * l));
    const unsigned pm = (unsigned)(P % m);
    for (unsigned x = 1; x < m; ++x)
      if ((pm * x) % m == 1u) {
        p->w[i] = (int)x;
        p->fw[i] = (float)x;
        break;
      }
  }
  for (int l = 0; l < 4; ++l) p->M[l] = (unsigned)(M >> (32 * l));
  return k;
}

namespace crtw {

constexpr int kParts = 6;   // 14-bit parts of a fixed-point row value (|F| <= 2^84)

// CRT digit weight of modulus t in the plan of the first k moduli: w_t = (M / m_t)^-1 mod m_t,
// M = m_0 ... m_{k-1}, the value plan() stores in w[t] (checked against it on the host), formed
// from small products only.
ZF_HD inline int digit_weight(int t, int k) {
  const int m = modulus(t);
  int p = 1 % m;
  for (int s = 0; s < k; ++s)
    if (s != t) p = (p * (modulus(s) % m)) % m;
  for (int x = 1; x < m; ++x)
    if ((p * x) % m == 1) return x;
  return 0;
}

// The six signed 14-bit parts of F (|F| <= 2^84), as floats: F = sum_k a_k 2^(14k).
ZF_HD inline void parts(unsigned long long mag_hi, unsigned long long mag_lo, bool neg, float (&a)[kParts]) {
  const float sg = neg ? -1.0f : 1.0f;
  for (int k = 0; k < kParts; ++k) {
    const int sh = 14 * k;
    unsigned long long v;
    if (sh + 14 <= 64)
      v = mag_lo >> sh;
    else if (sh >= 64)
      v = mag_hi >> (sh - 64);
    else
      v = (mag_lo >> sh) | (mag_hi << (64 - sh));
    a[k] = sg * (crt_bits_f(0x4B000000u | (unsigned)(v & 0x3FFFu)) - 8388608.0f);
  }
}

// Residue of F modulo m from its six parts: x = sum_k a_k (2^(14k) mod m) has |x / m| < 6 2^13, below
// 2^24 (exact in FP32); crt_residue_f's one reduction then errs by less than 0.0059 in the quotient, so
// |r| <= m (1/2 + 0.0059) < 129 for m <= 255, |r| <= 128 (m = 256: exact quotient).
ZF_HD inline float residue_f(const float (&a)[kParts], int m) {
  const float fm = (float)m;
  float x = a[kParts - 1] * (float)crt_pow2_sym(m, 14 * (kParts - 1));
  for (int k = kParts - 2; k >= 1; --k) x = fmaf(a[k], (float)crt_pow2_sym(m, 14 * k), x);
  x += a[0];
  return fmaf(-fm, crt_rint(x * (1.0f / fm)), x);
}

// sum_t y_t P_t per 32-bit limb (each limb sum below 2^47) and sum_t y_t / m_t in FP32 (error far
// below 1/4 for 24 terms); C = sum_t y_t P_t - q M modulo 2^192, exact while |C| < M / 4 < 2^183.
struct Acc {
  unsigned long long L[kLimbs];
  float S;
  ZF_HD void clear() {
    for (int l = 0; l < kLimbs; ++l) L[l] = 0ull;
    S = 0.0f;
  }
  // A sum y of CRT digits of modulus t (see CrtAcc::add_y): below 2^10, so every limb sum stays
  // below 2^47 over 24 moduli.
  ZF_HD void add_y(const Plan& p, int t, unsigned y) {
    S = fmaf(crt_u2f(y), p.inv[t], S);
    for (int l = 0; l < kLimbs; ++l) L[l] += (unsigned long long)y * p.P[t][l];
  }
  // C 2^sc in FP64, rounded once.  With a non-zero top word the magnitude is at least 2^128, so its
  // 53 leading bits lie in the top two words and the lowest word only decides the sticky bit (folded
  // into the lowest bit of the middle word, far below the rounding position).
  ZF_HD double value(const Plan& p, int sc) const {
    const long long q = crt_rint_i(S);
    unsigned l[kLimbs];
    long long carry = 0;
    for (int k = 0; k < kLimbs; ++k) {
      const long long t = (long long)L[k] - q * (long long)p.M[k] + carry;
      l[k] = (unsigned)t;
      carry = t >> 32;
    }
    unsigned long long w0 = ((unsigned long long)l[1] << 32) | l[0], w1 = ((unsigned long long)l[3] << 32) | l[2],
                       w2 = ((unsigned long long)l[5] << 32) | l[4];
    const bool neg = (l[5] >> 31) != 0u;
    if (neg) {
      w0 = ~w0 + 1ull;
      const unsigned long long c1 = w0 == 0ull ? 1ull : 0ull;
      w1 = ~w1 + c1;
      const unsigned long long c2 = (c1 && w1 == 0ull) ? 1ull : 0ull;
      w2 = ~w2 + c2;
    }
    if (w2 != 0ull) return crt_to_double(w2, w1 | (w0 != 0ull ? 1ull : 0ull), neg, 64 + sc);
    return crt_to_double(w1, w0, neg, sc);
  }
};

}  // namespace crtw
}  // namespace zf
