// The reconstruction over digits that no product wrote: for every moduli count and bytes at their ends, the value must
// not depend on what lies past the -q M table.
#include <cstdio>
#include <vector>

#include "crt_combine.h"

using namespace zf;

template <int SH>
static double value(const CrtCombine& c, const unsigned* bytes, const unsigned* qtab) {
  constexpr int Q = crt_shape_quads(SH), NB = crt_shape_bytes(SH), L = crt_shape_limbs(SH);
  unsigned d[Q] = {};
  for (int t = 0; t < c.nmod; ++t) d[t / 4] |= bytes[t] << (8 * (t % 4));
  return crt_combine_value<Q, NB, L>(c, d, qtab, crtw::kLimbs, 0);
}

static double dispatch(const CrtCombine& c, const unsigned* y, const unsigned* q) {
  switch (c.shape) {
    case 0: return value<0>(c, y, q);
    case 1: return value<1>(c, y, q);
    case 2: return value<2>(c, y, q);
    case 3: return value<3>(c, y, q);
    case 4: return value<4>(c, y, q);
    case 5: return value<5>(c, y, q);
    default: return value<6>(c, y, q);
  }
}

int main() {
  long long n = 0, bad = 0;
  unsigned long long s = 0x9E3779B97F4A7C15ull;
  for (int k = 1; k <= crtw::kMax; ++k) {
    const CrtCombine* c = crt_combine(k);
    if (!c) return 1;
    // the table, then words that differ between the two evaluations
    const size_t rows = sizeof(c->qM) / sizeof(c->qM[0]), words = rows * crtw::kLimbs;
    std::vector<unsigned> a(&c->qM[0][0], &c->qM[0][0] + words), b;
    a.resize(words + 64 * crtw::kLimbs, 0x13579BDFu);
    b = a;
    for (size_t w = words; w < b.size(); ++w) b[w] = ~a[w];
    for (int trial = 0; trial < 2000; ++trial) {
      unsigned y[crtw::kMax];
      for (int t = 0; t < crtw::kMax; ++t) {
        s ^= s << 13, s ^= s >> 7, s ^= s << 17;
        y[t] = trial == 0 ? 255u : trial == 1 ? 0u : trial % 2 ? (unsigned)(s & 0xFFu) : 224u | (unsigned)(s & 31u);
      }
      const double va = dispatch(*c, y, a.data()), vb = dispatch(*c, y, b.data());
      bad += memcmp(&va, &vb, sizeof(va)) != 0;
      ++n;
    }
  }
  printf("%lld checks, %lld bad\n", n, bad);
  return bad ? 1 : 0;
}
