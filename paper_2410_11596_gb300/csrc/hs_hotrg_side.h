// The choice between the two isometries of a HOTRG step (plain C++ on the host, so that
// a host test covers the solver's failures).
#pragma once

namespace hs {

// Side (0: left, 1: right) with the smaller discarded weight, ties left, among
// those whose two parity blocks were diagonalised: info[0..1] are the solver's statuses of
// the left Gram matrix's blocks, info[2..3] of the right one's. -1 if neither was.
// (A failed side's eigenvalues, and with them its discarded weight, mean nothing.)
inline int hotrg_side(const int info[4], double discarded_left, double discarded_right) {
  const bool left = info[0] == 0 && info[1] == 0, right = info[2] == 0 && info[3] == 0;
  if (!left && !right) return -1;
  if (left != right) return left ? 0 : 1;
  return discarded_left <= discarded_right ? 0 : 1;
}

}  // namespace hs
