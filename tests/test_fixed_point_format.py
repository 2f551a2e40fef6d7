"""The fixed-point format of the screened step's entries (csrc/fixed_point.h),
over table sizes up to those that nearly fill the word: whatever entry (of the
range, or 0 for one out of it) and difference meet, the sum modulo 2^32 lies in
[lo, hi] only if the exact sum does."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "fixed_point.h"
using namespace vcsgc;

static int checked = 0;

// sums of entries at both ends of the range, and of 0, with differences up to dmax
static bool sound(const FixedFormat& f, int K, double h, double dmax) {
  const long long d = 4 * (long long)std::lrint(dmax / h * std::ldexp(1.0, f.bits));
  const long long entries[] = {0, f.lo, f.lo + 4, f.hi - (K - 1), f.hi - (K - 1) - 4};
  const long long steps[] = {-d, -d + 4, -d / 2, -4, 0, 4, d / 2, d - 4, d};
  for (long long e : entries)
    for (int t = 0; t < K; ++t)
      for (long long s : steps) {
        const long long exact = e + t + s;
        const uint32_t word = (uint32_t)(e + t) + (uint32_t)s;
        const bool in = word >= f.lo && word <= f.hi, want = exact >= f.lo && exact <= f.hi;
        if (in != want || (e == 0 && in)) return false;
        ++checked;
      }
  return true;
}

int main() {
  int bad = 0, old_bad = 0, formats = 0;
  for (int K = 3; K <= 4; ++K)
    for (int n : {200, 500, 900, 1000, 1020, 1022, 1023, 2000, 4090, 4095, 5000, 8000, 8190})
      for (double d : {0.5, 3.0, 20.0, 24.0, 60.0, 150.0}) {  // largest difference, in intervals
        const double h = 0.013, lo = 0.2 * n * h, hi = n * h * (1.0 - 1e-6), dmax = d * h;
        const FixedFormat f = fixed_format(K, n, h, lo, hi, dmax);
        if (f.bits) {
          ++formats;
          bad += !sound(f, K, h, dmax);
          bad += (double)(n + 1) * std::ldexp(1.0, f.bits) > 1073741823.0;
        }
        // the largest number of bits that fits the grid, whatever the differences
        int bits = 23;
        while ((double)(n + 1) * std::ldexp(1.0, bits) > 1073741823.0) --bits;
        const double s = std::ldexp(1.0, bits) / h;
        const FixedFormat g{bits, (uint32_t)std::ceil(lo * s) << 2, (uint32_t)std::floor(hi * s) << 2 | (uint32_t)(K - 1)};
        if (dmax < 0.999 * lo) old_bad += !sound(g, K, h, dmax);
      }
  std::printf("%d %d %d %d\n", bad, old_bad, formats, checked);
  return 0;
}
"""


@pytest.fixture(scope="module")
def counts(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_1012_5082_gb300", "csrc"), str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    return [int(v) for v in subprocess.run([str(d / "t")], capture_output=True, text=True).stdout.split()]


def test_sums_leave_the_range_with_the_argument(counts):
    bad, _, formats, checked = counts
    assert bad == 0 and formats > 100 and checked > 10000


def test_the_largest_format_would_not_do(counts):
    """The check sees the wrap-around: with as many bits as the grid allows, some
    tables have sums that come round into the range."""
    assert counts[1] > 0
