// The reconstruction of a CRT product in 32-bit integer operations: bytes of the digits against bytes of the
// weights (four-way byte dot products), shared by the host planner and the kernels of k_crt.cu.  Plain C++
// outside nvcc, so the arithmetic can be checked on the host.
//
// T = sum_t y_t P_t (y_t the digits, P_t = M / m_t) equals C + q M with |C| < M / 4 and q the integer nearest
// sum_t y_t / m_t.  Byte b of the P_t gives t_b = sum_t y_t P_t[b] < 2^21 by one dot product per four moduli;
// q follows from sum_t y_t r_t with r_t = round(2^16 / m_t) (off by at most 24 * 255 / 2 in 2^16, below
// 1/20, where 1/4 is allowed); C = T - q M modulo 2^(32 limbs), with -q M from a table.
#pragma once
#include "crt_wide.h"

namespace zf {

// Rows of the -q M table.  Digits of a product give q <= 24; a row for every q that any bytes at all can give (at most
// 30, crt_combine_make checks it) keeps the index in the table where a product gave up and left its digits unwritten.
constexpr int kCrtQRows = 32;

// Constants for the first nmod moduli.  Moduli 4 i ... 4 i + 3 share a word (modulus 4 i in the lowest byte).
struct CrtCombine {
  int nmod;
  int shape;                                      // index of the kernels' (quads, bytes, limbs), crt_shape
  unsigned W[4 * crtw::kLimbs][crtw::kMax / 4];   // byte b of P_t
  unsigned R[crtw::kMax / 4];                     // round(2^16 / m_t) - 256
  unsigned qM[kCrtQRows][crtw::kLimbs];           // -q M modulo 2^192
  float fw[32];                                   // digit weights (M / m_t)^-1 mod m_t, for the products' epilogue
};

// The kernels' instantiations: words of four moduli, bytes of the P_t, limbs that hold |C| < M / 4 and its
// sign.  P_t < 2^55.9 for up to 8 moduli, 2^87.1 for 12, 2^94.8 for 13, 2^110.2 for 15, 2^117.8 for 16, 2^148
// for 20 and 2^177.4 for 24 (checked by crt_combine).
constexpr int kCrtShapes = 7;
ZF_HD constexpr int crt_shape(int k) {
  return k <= 8 ? 0 : k <= 12 ? 1 : k <= 13 ? 2 : k <= 15 ? 3 : k <= 16 ? 4 : k <= 20 ? 5 : 6;
}
ZF_HD constexpr int crt_shape_quads(int s) { return s == 0 ? 2 : s == 1 ? 3 : s <= 4 ? 4 : s; }
ZF_HD constexpr int crt_shape_bytes(int s) { return s == 0 ? 8 : s <= 2 ? 12 : s == 3 ? 14 : s == 4 ? 16 : s == 5 ? 20 : 24; }
ZF_HD constexpr int crt_shape_limbs(int s) { return s == 0 ? 2 : s == 1 ? 3 : s <= 4 ? 4 : s; }

ZF_HD inline unsigned crt_dp4(unsigned a, unsigned b, unsigned c) {
#ifdef __CUDA_ARCH__
  return __dp4a(a, b, c);
#else
  for (int i = 0; i < 4; ++i) c += ((a >> (8 * i)) & 0xFFu) * ((b >> (8 * i)) & 0xFFu);
  return c;
#endif
}
ZF_HD inline int crt_clz32(unsigned x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
ZF_HD inline unsigned crt_shl(unsigned lo, unsigned hi, int s) {  // the upper word of (hi : lo) << s, s < 32
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, s);
#else
  return s ? (hi << s) | (lo >> (32 - s)) : hi;
#endif
}

// (-1)^neg |x| 2^sc for the magnitude x in L words (lowest first), rounded once to the nearest double (ties
// to even); integer operations only (crt.h's crt_to_double says why).
template <int L>
ZF_HD inline double crt_words_to_double(unsigned (&x)[L], bool neg, int sc) {
  int e = 32 * L - 1 + sc;
  unsigned rest = 0u;  // words below the top three: only whether they are zero counts
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int s = 1; s < L; ++s)
    if (x[L - 1] == 0u) {
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
      for (int k = L - 1; k > 0; --k) x[k] = x[k - 1];
      x[0] = 0u;
      e -= 32;
    }
  const unsigned a0 = x[L - 1], b0 = x[L - 2], c0 = L > 2 ? x[L > 2 ? L - 3 : 0] : 0u;
  if (a0 == 0u) return 0.0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int k = 0; k < L - 3; ++k) rest |= x[k];
  const int lz = crt_clz32(a0);
  e -= lz;
  const unsigned a = crt_shl(b0, a0, lz), b = crt_shl(c0, b0, lz), c = (c0 << lz) | rest;
  const int be = e + 1023;
  if (be <= 0 || be >= 2046)  // near the ends of the range: crt.h's careful form (c as the sticky bit)
    return crt_to_double(((unsigned long long)a << 32) | b, c ? 1ull : 0ull, neg, e - 127);
  // 53 bits: a and the upper 21 of b, with the leading one adding to the exponent field
  const unsigned lo = (a << 21) | (b >> 11), hi = (a >> 11) + ((unsigned)(be - 1) << 20) + (neg ? 0x80000000u : 0u);
  const unsigned up = ((b >> 10) & 1u) & (((b & 0x3FFu) | c) != 0u ? 1u : (lo & 1u));
  const unsigned long long r = (((unsigned long long)hi << 32) | lo) + up;
  return crt_bits_d(r);
}

// C 2^sc from the digit words d (word i: the digits of moduli 4 i ... 4 i + 3; 0 past nmod) and a row of the
// qM table for every q (stride words apart).
template <int Q, int NB, int L>
ZF_HD inline double crt_combine_value(const CrtCombine& p, const unsigned (&d)[Q], const unsigned* qtab, int stride,
                                      int sc) {
  unsigned s1 = 0u, s2 = 32768u;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < Q; ++i) {
    s1 = crt_dp4(d[i], 0x01010101u, s1);
    s2 = crt_dp4(d[i], p.R[i], s2);
  }
  const unsigned q = (s1 * 256u + s2) >> 16;
  const unsigned* qm = qtab + q * stride;
  unsigned x[L];
  unsigned long long acc = 0ull;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int w = 0; w < L; ++w) {
    unsigned t[4] = {0u, 0u, 0u, 0u};
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int b = 0; b < 4; ++b)
      if (4 * w + b < NB)
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int i = 0; i < Q; ++i) t[b] = crt_dp4(d[i], p.W[4 * w + b][i], t[b]);
    acc += (unsigned long long)(t[0] + (t[1] << 8)) + ((unsigned long long)(t[2] + (t[3] << 8)) << 16) + qm[w];
    x[w] = (unsigned)acc;
    acc >>= 32;
  }
  const bool neg = (x[L - 1] >> 31) != 0u;
  if (neg) {
    unsigned long long c = 1ull;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int w = 0; w < L; ++w) {
      c += (unsigned)~x[w];
      x[w] = (unsigned)c;
      c >>= 32;
    }
  }
  return crt_words_to_double<L>(x, neg, sc);
}

// The constants of the first k moduli (1 <= k <= crtw::kMax); false when a P_t does not fit its shape, or a q the table.
inline bool crt_combine_make(int k, CrtCombine* c) {
  crtw::Plan p;
  double bits = 0.0;  // as the planners sum them: plan() takes exactly k
  for (int t = 0; t + 1 < k; ++t) bits += log2((double)crtw::modulus(t));
  if (crtw::plan(bits, &p) != k) return false;
  memset(c, 0, sizeof(*c));
  c->nmod = k;
  c->shape = crt_shape(k);
  for (int t = 0; t < k; ++t) {
    const int q = t / 4, sh = 8 * (t % 4);
    c->fw[t] = p.fw[t];
    c->R[q] |= (unsigned)(((1 << 17) / p.m[t] + 1) / 2 - 256) << sh;
    for (int b = 0; b < 4 * crtw::kLimbs; ++b) {
      const unsigned v = (p.P[t][b / 4] >> (8 * (b % 4))) & 0xFFu;
      if (v && b >= crt_shape_bytes(c->shape)) return false;
      c->W[b][q] |= v << sh;
    }
  }
  unsigned qmax = 32768u;  // 2^16 q of digits that are all 255
  for (int t = 0; t < k; ++t) qmax += 255u * (256u + ((c->R[t / 4] >> (8 * (t % 4))) & 0xFFu));
  if ((qmax >> 16) >= (unsigned)kCrtQRows) return false;
  for (int q = 0; q < kCrtQRows; ++q) {
    unsigned long long mul = 0ull, neg = 1ull;
    for (int l = 0; l < crtw::kLimbs; ++l) {
      mul += (unsigned long long)q * p.M[l];
      neg += (unsigned)~(unsigned)mul;
      c->qM[q][l] = (unsigned)neg;
      mul >>= 32;
      neg >>= 32;
    }
  }
  return true;
}

// The moduli count whose product exceeds 2^bits (the rule of crt_plan and crtw::plan); 0 if all do not.
inline int crt_count(double bits) {
  double lb = 0.0;
  int k = 0;
  while (k < crtw::kMax && lb <= bits) lb += log2((double)crtw::modulus(k++));
  return lb <= bits ? 0 : k;
}

// The constants of k moduli, made once per process (they depend on k alone).
inline const CrtCombine* crt_combine(int k) {
  struct All {
    CrtCombine c[crtw::kMax + 1];
    bool ok[crtw::kMax + 1];
    All() {
      for (int k = 1; k <= crtw::kMax; ++k) ok[k] = crt_combine_make(k, &c[k]);
    }
  };
  static const All all;
  return k >= 1 && k <= crtw::kMax && all.ok[k] ? &all.c[k] : nullptr;
}

}  // namespace zf
