// Host check of the digit slices of an FP64 row and of the fixed-point result
// (csrc/hs_bits.cuh): the digits rebuild the fixed-point value, which is within
// half a unit of the number, and the 64-bit sum converts like the FPU does.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../paper_2410_11596_gb300/csrc/hs_bits.cuh"

using namespace hs;

int main() {
  std::mt19937_64 g(1);
  long bad = 0;
  for (long t = 0; t < 2000000; ++t) {
    const int emax = 100 + (int)(g() % 1946);
    // exponents from emax down to 80 below it, subnormals and zeros, and the largest and smallest mantissas
    const int ef = t % 11 == 0 ? 0 : emax - (int)(g() % 80);
    unsigned long long m = g() & 0xFFFFFFFFFFFFFull;
    if (t % 13 == 0) m = 0xFFFFFFFFFFFFFull;
    if (t % 17 == 0) m = 0;
    const double x = f64_from_bits((g() & (1ull << 63)) | ((unsigned long long)ef << 52) | m);
    const long long X = slice_fixed(f64_bits(x), emax), Y = slice_bias(X);
    long long back = 0;
    for (int i = 1; i <= 7; ++i) {
      const int d = slice_digit(Y, i);
      bad += d < -128 || d > (i == 1 ? 128 : 127);
      back = back * 256 + d;
    }
    bad += back != X;
    const long double unit = ldexpl(1.0L, emax - 1022 - 55);
    bad += fabsl((long double)X * unit - (long double)x) > 0.5L * unit;
    const long long J = (long long)g() >> (1 + g() % 62);
    const int s = (int)(g() % 1200) - 600;
    const double r = std::ldexp((double)J, s);
    bad += J == 0 ? fixed_to_f64(J, s) != 0 : fixed_to_f64(J, s) != f64_bits(r);
  }
  const long long top = 0x7FFFFFFFFFFFFFFFll;
  bad += fixed_to_f64(top, 0) != f64_bits((double)top) || fixed_to_f64(-top, 0) != f64_bits(-(double)top);
  bad += fixed_to_f64(1, -900) != f64_bits(std::ldexp(1.0, -900));
  std::printf("bad %ld\n", bad);
  return bad ? 1 : 0;
}
