// Host check of the scaled entries and magnitudes behind the digit slices
// (csrc/hs_bits.cuh): powers of two against ldexp, magnitudes against the number.
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_2410_11596_gb300/csrc/hs_bits.cuh"

using namespace hs;

static double e5m2(uint32_t v) { return v < 4 ? v * std::ldexp(1.0, -16) : std::ldexp(1.0 + (v & 3) / 4.0, (int)(v >> 2) - 15); }

int main() {
  std::mt19937_64 g(2);
  long bad = 0;
  for (long t = 0; t < 2000000; ++t) {
    const int emax = 100 + (int)(g() % 1946);
    int ef = t % 11 == 0 ? 0 : emax - (int)(g() % 80);
    unsigned long long m = g() & 0xFFFFFFFFFFFFFull;
    if (t % 13 == 0) m = 0xFFFFFFFFFFFFFull;
    if (t % 17 == 0) m = 0;
    const unsigned long long b = (g() & (1ull << 63)) | ((unsigned long long)ef << 52) | m;
    const double x = f64_from_bits(b), mag = std::ldexp(std::fabs(x), 1022 - emax);  // over the row's scale, < 1
    const uint32_t v = slice_mag8(b, emax);
    bad += v > 0x7B || (v == 0) != (x == 0.0);
    if (x != 0.0) {
      const double y = std::ldexp(e5m2(v), -15);
      bad += mag >= std::ldexp(1.0, -29) ? !(y <= mag && y >= 0.8 * mag) : y != std::ldexp(1.0, -29);
    }
    const float f = slice_magf(b, emax);
    bad += ef == 0 ? f > 1e-30f : !(f <= mag && f >= mag * (1 - std::ldexp(1.0, -20)));
    // powers of two
    const int adj = (int)(g() % 801) - 400;
    const double s = f64_from_bits(slice_scaled(b, adj));
    if (ef == 0) {
      bad += f64_bits(s) != b;
    } else if (ef + adj >= 0x7FF) {
      bad += !std::isinf(s) || std::signbit(s) != std::signbit(x);
    } else if (ef + adj <= 0) {
      bad += s == 0.0 || std::fabs(s) > std::ldexp(1.0, -1022) || std::signbit(s) != std::signbit(x);
    } else {
      bad += s != std::ldexp(x, adj);
    }
  }
  for (double x : {(double)INFINITY, -(double)INFINITY, 0.0, -0.0}) bad += slice_scaled(f64_bits(x), 37) != f64_bits(x);
  bad += !std::isnan(f64_from_bits(slice_scaled(f64_bits((double)NAN), -37)));
  std::printf("bad %ld\n", bad);
  return bad ? 1 : 0;
}
