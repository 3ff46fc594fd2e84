// Host check of the side a HOTRG step takes (csrc/hs_hotrg_side.h).
#include <cmath>
#include <cstdio>

#include "../paper_2410_11596_gb300/csrc/hs_hotrg_side.h"

int main() {
  int bad = 0;
  const double nan = std::nan("");
  for (int f = 0; f < 16; ++f) {
    const int info[4] = {f & 1, f & 2 ? 3 : 0, f & 4 ? -2 : 0, f & 8 ? 7 : 0};
    const bool left = !(f & 3), right = !(f & 12);
    const double w[4][2] = {{1.0, 2.0}, {2.0, 1.0}, {1.0, 1.0}, {left ? 1.0 : nan, right ? 2.0 : nan}};
    for (const auto& d : w) {
      const int want = left && right ? (d[0] <= d[1] ? 0 : 1) : left ? 0 : right ? 1 : -1;
      bad += hs::hotrg_side(info, d[0], d[1]) != want;
    }
  }
  std::printf("bad %d\n", bad);
  return bad ? 1 : 0;
}
