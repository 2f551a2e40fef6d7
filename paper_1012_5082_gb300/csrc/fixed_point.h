// Fixed-point format of the screened step's per-site entries (host side): an
// embedding argument x / h with `bits` fraction bits above two species bits, in
// an unsigned word.  A trial adds a shell's difference to an entry; the sum has
// to leave [lo, hi] whenever the argument does, also where it wraps around.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace vcsgc {

struct FixedFormat {
  int bits;         // 0: none
  uint32_t lo, hi;  // packed arguments of the screened range
};

// K species, n intervals of width h, arguments in [lo, hi], differences of at
// most dmax in size.
//  - An argument of the grid and one interval more fit in 30 bits.
//  - hi plus the largest difference stays below 2^32 (else it would come round
//    to 0 and up), and so does the other way 2^32 minus a difference stay above
//    hi: an entry out of range is stored as 0, and 0 less a difference wraps to
//    the top.  No difference alone reaches lo from 0.
//  - The rounding of an argument, 2 2^-bits intervals, stays within what a float
//    argument takes from interval j0 up: 4 (j0 + 2) 2^-24 intervals.
inline FixedFormat fixed_format(int K, int n, double h, double lo, double hi, double dmax) {
  FixedFormat f{0, 0u, 0u};
  if (!(dmax < 0.999 * lo)) return f;
  const int j0 = std::max(0, (int)std::floor(lo / h) - 1);
  for (int bits = 23; std::ldexp(1.0, 25 - bits) <= 4.0 * (j0 + 2) && bits > 0; --bits) {
    const double scale = std::ldexp(1.0, bits);
    if ((double)(n + 1) * scale > 1073741823.0) continue;
    const double top = 4.0 * std::floor(hi / h * scale) + (K - 1);
    if (4.0 * (std::ceil(dmax / h * scale) + 1.0) >= 4294967296.0 - top) continue;
    f.bits = bits;
    f.lo = (uint32_t)std::ceil(lo / h * scale) << 2;
    f.hi = (uint32_t)top;
    return f;
  }
  return f;
}

}  // namespace vcsgc
