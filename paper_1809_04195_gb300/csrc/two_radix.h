// Lengths that are a product of two radices with register butterflies: the radix set and the choice
// of a pair, shared by the kernels that select their radices at run time.
#pragma once

#include <algorithm>

namespace t2sh {

constexpr int kMaxRadix = 25;
// X(R) for every radix
#define T2SH_RADICES(X) X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(13) X(15) X(16) X(18) X(20) X(25)

constexpr int kRadix[] = {2, 3, 4, 5, 6, 8, 9, 10, 12, 13, 15, 16, 18, 20, 25};

// The pair of radices of a length: the most even one (fewest registers, every thread busy in both
// stages); among equals the larger first.  first_max bounds the first radix; four prefers a first
// radix that is a multiple of four (aligned chunks on the side of t).
inline bool two_radices(int n, int first_max, bool four, int* r0, int* r1) {
  int best = 1 << 30;
  for (int a : kRadix) {
    if (a > first_max || n % a) continue;
    for (int b : kRadix)
      if (a * b == n) {
        const int cost = 4 * std::max(a, b) + (four && a % 4 ? 8 : 0) + (a < b ? 1 : 0);
        if (cost < best) {
          best = cost;
          *r0 = a;
          *r1 = b;
        }
      }
  }
  return best < (1 << 30);
}

}  // namespace t2sh
