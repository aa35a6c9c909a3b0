// The running residue sums of a product's epilogue over up to 64 sub-chunks (N = 65536), two columns to a float, with the
// fold after every kCrtFoldSub of them: both columns' digits against integers, for runs of the largest residues of either
// sign, carries at their ends, and random sums.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "crt_wide.h"

using namespace zf;

static long long mod(long long a, long long m) { return ((a % m) + m) % m; }

int main() {
  srand(11);
  long long bad = 0, n = 0;
  for (int t = 0; t < crtw::kMax; ++t) {
    const int mi = crtw::modulus(t), top = mi / 2;
    const float m = (float)mi, inv = 1.0f / m;
    for (int trial = 0; trial < 3000; ++trial) {
      // column a: a prefix of extremes and zeros that leaves a carry, then extremes; column b: a small odd or even sum
      const int sa = trial & 1 ? 1 : -1, zeros = trial / 2 % 5, b0 = (trial / 10 % 9) - 4, kind = trial % 7;
      float p = 0.0f;
      long long s0 = 0, s1 = 0;
      for (int k = 0; k < 64; ++k) {
        long long a = k >= 16 - zeros && k < 16 ? 0 : sa * top, b = k == 0 ? b0 : 0;
        if (kind == 5) a = k % 2 ? sa * top : (rand() % 3 - 1) * top;
        if (kind == 6) a = rand() % (2 * top + 1) - top, b = rand() % (2 * top + 1) - top;
        if (trial / 3 % 4 == 0) {  // full-size sums of the same residues (an exact FP32 sum is at most 2^24)
          const long long q = rand() % (((1 << 24) - mi) / mi);
          a += (a < 0 ? -1 : 1) * q * mi;
        }
        const bool swap = trial % 3 == 2;
        const long long v0 = swap ? b : a, v1 = swap ? a : b;
        p = fmaf(crt_step((float)v1, m, inv), 4096.0f, p + crt_step((float)v0, m, inv));
        s0 += v0;
        s1 += v1;
        float r0, r1;
        crt_unpack2(p, &r0, &r1);
        bad += !(fabsf(r0) < 2048.0f) || !(fabsf(r1) < 2048.0f);
        bad += mod((long long)r0 - s0, mi) != 0 || mod((long long)r1 - s1, mi) != 0;
        const float w = (float)(1 + (trial * 31 + k) % (mi - 1));
        bad += (long long)crt_digit_sum(r0, m, inv, w) != mod(mod(s0, mi) * (long long)w, mi);
        bad += (long long)crt_digit_sum(r1, m, inv, w) != mod(mod(s1, mi) * (long long)w, mi);
        ++n;
        if (k % kCrtFoldSub == kCrtFoldSub - 1) p = fmaf(crt_step(r1, m, inv), 4096.0f, crt_step(r0, m, inv));
      }
    }
  }
  printf("%lld checks, %lld bad\n", n, bad);
  return bad ? 1 : 0;
}
