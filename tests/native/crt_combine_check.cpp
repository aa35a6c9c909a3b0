// The byte-wise reconstruction (crt_combine.h) against the limb sums of crt_wide.h, for every moduli count: the
// digits of products C at the ends of |C| < M / 4, near zero, at rounding ties, and random, as doubles bit for
// bit, over the whole exponent range.
#include <cstdio>
#include <cstdlib>

#include "crt_combine.h"

using namespace zf;

typedef unsigned Words[crtw::kLimbs];  // two's complement, lowest first

static unsigned long long rnd() {
  static unsigned long long s = 0x9E3779B97F4A7C15ull;
  s ^= s << 13, s ^= s >> 7, s ^= s << 17;
  return s;
}

static unsigned mod_words(const Words& c, unsigned m) {  // C mod m for the signed C
  const bool neg = c[crtw::kLimbs - 1] >> 31;
  unsigned long long carry = neg ? 1 : 0, r = 0;
  Words a;
  for (int l = 0; l < crtw::kLimbs; ++l) {
    carry += neg ? (unsigned)~c[l] : c[l];
    a[l] = (unsigned)carry;
    carry >>= 32;
  }
  for (int l = crtw::kLimbs - 1; l >= 0; --l) r = ((r << 32) | a[l]) % m;
  return (unsigned)(neg && r ? m - r : r);
}

template <int SH>
static double value(const CrtCombine& c, const unsigned (&y)[crtw::kMax], int sc) {
  constexpr int Q = crt_shape_quads(SH), NB = crt_shape_bytes(SH), L = crt_shape_limbs(SH);
  unsigned d[Q] = {};
  for (int t = 0; t < c.nmod; ++t) d[t / 4] |= y[t] << (8 * (t % 4));
  return crt_combine_value<Q, NB, L>(c, d, &c.qM[0][0], crtw::kLimbs, sc);
}

static double dispatch(const CrtCombine& c, const unsigned (&y)[crtw::kMax], int sc) {
  switch (c.shape) {
    case 0: return value<0>(c, y, sc);
    case 1: return value<1>(c, y, sc);
    case 2: return value<2>(c, y, sc);
    case 3: return value<3>(c, y, sc);
    case 4: return value<4>(c, y, sc);
    case 5: return value<5>(c, y, sc);
    default: return value<6>(c, y, sc);
  }
}

int main() {
  long long n = 0, bad = 0;
  for (int k = 1; k <= crtw::kMax; ++k) {
    const CrtCombine* c = crt_combine(k);
    crtw::Plan p;
    double bits = 0.0;
    for (int t = 0; t + 1 < k; ++t) bits += log2((double)crtw::modulus(t));
    if (!c || crtw::plan(bits, &p) != k || crt_count(bits) != k) {
      printf("no plan for %d\n", k);
      return 1;
    }
    bits += log2((double)crtw::modulus(k - 1));
    for (int trial = 0; trial < 60000; ++trial) {
      // |C| < M / 4: `top` bits of magnitude, patterned low bits
      const int most = (int)floor(bits) - 3;
      const int top = trial % 3 == 0 ? most : 1 + (int)(rnd() % (most > 0 ? most : 1));
      Words w = {};
      if (most > 0)
        for (int b = 0; b < top; ++b) {
          const int kind = trial % 5;
          const bool bit = b == top - 1                    ? true
                           : kind == 0                     ? true                        // 2^top - 1
                           : kind == 1                     ? b == top - 54               // a tie below 53 bits
                           : kind == 2                     ? b == top - 54 || b == 0     // just above a tie
                           : kind == 3 && b > top - 54     ? true                        // carries through the mantissa
                                                           : rnd() & 1;
          if (bit) w[b / 32] |= 1u << (b % 32);
        }
      if (rnd() & 1) {  // negative
        unsigned long long carry = 1;
        for (int l = 0; l < crtw::kLimbs; ++l) {
          carry += (unsigned)~w[l];
          w[l] = (unsigned)carry;
          carry >>= 32;
        }
      }
      unsigned y[crtw::kMax] = {};
      crtw::Acc acc;
      acc.clear();
      for (int t = 0; t < k; ++t) {
        y[t] = mod_words(w, (unsigned)p.m[t]) * (unsigned)p.w[t] % (unsigned)p.m[t];
        acc.add_y(p, t, y[t]);
      }
      const int sc = trial % 7 == 0 ? -1074 - (int)(rnd() % 200) : trial % 7 == 1 ? 900 - (int)(rnd() % 300) : -(int)(rnd() % 200);
      const double a = acc.value(p, sc), b = dispatch(*c, y, sc);
      bad += memcmp(&a, &b, 8) != 0;
      ++n;
    }
  }
  printf("%lld checks, %lld bad\n", n, bad);
  return bad ? 1 : 0;
}
