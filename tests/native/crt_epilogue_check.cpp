// The residue steps of the product's epilogue against integers: for every modulus, sub-chunk sums at the
// ends of their range and in between, two columns to a float over kCrtFoldSub steps, and the digit.
#include <cstdio>
#include <cstdlib>

#include "crt_wide.h"

using namespace zf;

static long long mod(long long a, long long m) { return ((a % m) + m) % m; }

int main() {
  srand(7);
  long long bad = 0, n = 0;
  for (int t = 0; t < crtw::kMax; ++t) {
    const int mi = crtw::modulus(t);
    const float m = (float)mi, inv = 1.0f / m;
    for (int trial = 0; trial < 4000; ++trial) {
      float p = 0.0f;
      long long s0 = 0, s1 = 0;
      const int w = 1 + (trial * 37 + rand()) % (mi - 1);
      for (int k = 0; k < kCrtFoldSub; ++k) {
        long long v[2];
        for (int c = 0; c < 2; ++c) {
          const long long r = ((long long)rand() << 8) ^ rand();
          // the range's ends, multiples and half multiples of m (ties of the quotient), and random sums
          v[c] = trial % 4 == 0   ? (r & 1 ? (1 << 24) : -(1 << 24)) + (trial / 4 % 512) * (r & 1 ? -1 : 1)
                 : trial % 4 == 1 ? (r % 60000) * mi
                 : trial % 4 == 2 ? (r % 60000) * mi + mi / 2 + (r >> 20) % 2
                                  : r % (1 << 24);
          if (trial % 8 >= 4) v[c] = -v[c];
          if (v[c] > (1 << 24)) v[c] = 1 << 24;
          if (v[c] < -(1 << 24)) v[c] = -(1 << 24);
        }
        const float r0 = crt_step((float)v[0], m, inv), r1 = crt_step((float)v[1], m, inv);
        bad += !(fabsf(r0) <= 0.507f * m + 0.5f) || !(fabsf(r1) <= 0.507f * m + 0.5f);
        bad += mod((long long)r0 - v[0], mi) != 0 || mod((long long)r1 - v[1], mi) != 0;
        p = fmaf(r1, 4096.0f, p + r0);
        s0 += v[0];
        s1 += v[1];
      }
      float q0, q1;
      crt_unpack2(p, &q0, &q1);
      bad += !(fabsf(q0) < 2048.0f) || !(fabsf(q1) < 2048.0f);
      bad += (long long)crt_digit_sum(q0, m, inv, (float)w) != mod(mod(s0, mi) * w, mi);
      bad += (long long)crt_digit_sum(q1, m, inv, (float)w) != mod(mod(s1, mi) * w, mi);
      n += 2;
    }
    // every sum the digit can be asked for
    for (int s = -2047; s <= 2047; ++s)
      for (int w = 1; w < mi; w += 1 + w / 8) {
        bad += (long long)crt_digit_sum((float)s, m, inv, (float)w) != mod((long long)s * w, mi);
        ++n;
      }
  }
  printf("%lld checks, %lld bad\n", n, bad);
  return bad ? 1 : 0;
}
