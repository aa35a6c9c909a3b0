// Host check of the residue step of the operand kernels (crt.h: crt_part_f, crt_residue_step): congruent to the
// exact value and within 128 of zero for every modulus, with four, five and six parts, at the ends of their ranges
// and at random.
#include <stdio.h>

#include <random>

#include "../../paper_2404_19163_gb300/csrc/crt_wide.h"

using namespace zf;

template <int NP>
static long check(std::mt19937_64& rng, int bits) {
  long fails = 0;
  for (int it = 0; it < 40000; ++it) {
    unsigned __int128 mag = ((unsigned __int128)rng() << 64) | rng();
    mag >>= 128 - bits;                                             // random below 2^bits
    if (it % 8 == 1) mag >>= rng() % bits;                          // of any length
    if (it % 8 == 2) mag = ((unsigned __int128)1 << bits) - it % 5;  // at the end (|F| <= 2^bits)
    if (it % 8 == 3) mag = it % 300;
    const bool neg = it & 1;
    float a[NP];
    for (int k = 0; k < NP; ++k) a[k] = crt_part_f((unsigned)(mag >> (14 * k)) & 0x3FFFu, neg ? 0x80000000u : 0u);
    for (int t = 0; t < crtw::kMax; ++t) {
      const int m = crtw::modulus(t);
      const float r = crt_residue_step<NP>(a, m);
      const int ri = (int)r, want = (int)(mag % (unsigned)m);
      const int got = ((neg ? -ri : ri) % m + m) % m;
      if ((float)ri != r || ri > kCrtMaxResidue || ri < -kCrtMaxResidue || got != want) ++fails;
    }
  }
  return fails;
}

int main() {
  std::mt19937_64 rng(11);
  const long f4 = check<4>(rng, 55), f5 = check<5>(rng, 62), f6 = check<6>(rng, 83);
  printf("fails %ld\n", f4 + f5 + f6);
  return f4 + f5 + f6 ? 1 : 0;
}
