// sum_f32_in_f64 against the FP64 adds it stands for, bit for bit.
#include <cstdio>
#include <random>

#include "../paper_2410_11596_gb300/csrc/hs_bits.cuh"

int main() {
  std::mt19937_64 rng(7);
  long long bad = 0, n = 0;
  for (int spread : {0, 1, 24, 25, 26, 40, 253}) {
    for (int rep = 0; rep < 200000; ++rep) {
      float x[16];
      const int k = 1 + (int)(rng() % 16);
      const int lo = spread > 252 ? 0 : (int)(rng() % (254 - spread));  // 0: subnormals and zeros
      double want = 0.0;
      for (int i = 0; i < k; ++i) {
        uint32_t m = (uint32_t)rng() & 0x7FFFFFu;
        if (rng() % 4 == 0) m = rng() % 2 ? 0x7FFFFFu : 0u;
        uint32_t u = (uint32_t)(lo + rng() % (spread + 1)) << 23 | m | ((uint32_t)rng() & 0x80000000u);
        if (rng() % 16 == 0) u &= 0x80000000u;  // signed zero
        if (rng() % 4000 == 0) u = (u & 0x80000000u) | 0x7F800000u;
        std::memcpy(&x[i], &u, 4);
        if (i > 0 && rng() % 8 == 0) x[i] = -x[i - 1];
        want += (double)x[i];
      }
      const double got = hs::sum_f32_in_f64<16>(x, k);
      ++n;
      if (hs::f64_bits(got) != hs::f64_bits(want) && !(got != got && want != want)) ++bad;
    }
  }
  std::printf("%lld of %lld sums differ\n", bad, n);
  return bad != 0;
}
