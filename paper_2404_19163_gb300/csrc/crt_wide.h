// The moduli of the residue products and their plans: crt.h's sixteen moduli and eight more, up to 24 pairwise coprime
// ones (M about 2^184.6, six 32-bit limbs) for fixed-point rows of up to 83 bits.  A plan takes the first k.  Every modulus is
// at most 256, so the residues, the K-chunk length (1024) and the FP32 reductions are those of crt.h.
//
// Used by k_ozmod.cu (residues), the products' epilogue and, through crt_combine.h, the reconstruction of k_crt.cu.
#pragma once
#include "crt.h"

namespace zf {
namespace crtw {

constexpr int kMax = 24;    // moduli
constexpr int kLimbs = 6;   // 32-bit limbs of M and of the digit sums

// crt.h's sixteen moduli, then the next primes below 193 (coprime to all of them).
ZF_HD constexpr int modulus(int i) {
  if (i < kCrtMax) return crt_modulus(i);
  switch (i) {
    case 16: return 191;
    case 17: return 181;
    case 18: return 179;
    case 19: return 173;
    case 20: return 167;
    case 21: return 163;
    case 22: return 157;
    case 23: return 151;
    default: return 1;
  }
}

// The first nmod moduli: P_i = M / m_i, digit weights w_i = P_i^-1 mod m_i.
struct Plan {
  int nmod;
  int m[kMax];
  int w[kMax];
  float inv[kMax], fm[kMax], fw[kMax];
  unsigned P[kMax][kLimbs];
  unsigned M[kLimbs];
};

// The moduli count that makes M exceed 2^bits (0 if all 24 do not), with the constants.  M and
// M / m_i are formed in 32-bit limbs (products and quotients by small integers only).
inline int plan(double bits, Plan* p) {
  unsigned M[kLimbs + 1] = {1u};
  int k = 0;
  double lb = 0.0;
  while (k < kMax && lb <= bits) {
    const unsigned m = (unsigned)modulus(k);
    unsigned long long c = 0;
    for (int l = 0; l <= kLimbs; ++l) {
      const unsigned long long t = (unsigned long long)M[l] * m + c;
      M[l] = (unsigned)t;
      c = t >> 32;
    }
    lb += log2((double)m);
    ++k;
  }
  if (lb <= bits || M[kLimbs] != 0u) return 0;
  p->nmod = k;
  for (int l = 0; l < kLimbs; ++l) p->M[l] = M[l];
  for (int i = 0; i < kMax; ++i) {
    const unsigned m = i < k ? (unsigned)modulus(i) : 1u;
    p->m[i] = (int)m;
    p->inv[i] = 1.0f / (float)m;
    p->fm[i] = (float)m;
    p->w[i] = 0;
    p->fw[i] = 0.0f;
    for (int l = 0; l < kLimbs; ++l) p->P[i][l] = 0u;
    if (i >= k) continue;
    // P = M / m from the top limb down; the remainder of M / m is 0, and P mod m follows from P's limbs
    unsigned long long rem = 0;
    for (int l = kLimbs - 1; l >= 0; --l) {
      const unsigned long long cur = (rem << 32) | M[l];
      p->P[i][l] = (unsigned)(cur / m);
      rem = cur % m;
    }
    unsigned long long pm = 0;
    for (int l = kLimbs - 1; l >= 0; --l) pm = ((pm << 32) | p->P[i][l]) % m;
    for (unsigned x = 1; x < m; ++x)
      if ((pm * x) % m == 1u) {
        p->w[i] = (int)x;
        p->fw[i] = (float)x;
        break;
      }
  }
  return k;
}

}  // namespace crtw
}  // namespace zf

#ifndef __CUDACC__
#include "crt_reference.h"  // the host checks' reference forms
#endif
