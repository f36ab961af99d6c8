"""The stored-weight walk's 32-bit byte offsets at the ends of the range it is taken for, in a
constant expression (where a signed overflow does not compile), against 64-bit arithmetic."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1509_02468_gb300", "csrc")

SOURCE = """
#include "bf_index.h"
// weight of plane f, `shift` samples from pixel i: both routes
constexpr bool right(long long n, long long i, int f0, int f, long long shift, int es) {
  return bf_tap_offset(bf_base_offset((unsigned)i, (unsigned)f0, (unsigned)n, (unsigned)es),
                       (f - f0) * (int)n + (int)shift, es) ==
         (unsigned long long)((f * n + i + shift) * es);
}
// every plane, from the first and the last pixel: 3 rows and columns back where that lies in the
// planes; and the strip's pixels past the image, which are not read
constexpr bool ends(long long n, long long nx, int f0, int es) {
  if (!bf_tap_offset_fits(n, nx, f0, es)) return false;
  for (int f = 0; f < 24; ++f) {
    if (!right(n, n - 1, f0, f, 0, es) || !right(n, 0, f0, f, 0, es)) return false;
    if (3 * nx + 3 < n && (!right(n, n - 1, f0, f, -3 * nx - 3, es) || !right(n, 3 * nx + 3, f0, f, -3 * nx - 3, es)))
      return false;
    if (bf_tap_offset(0, (f - f0) * (int)n + (int)(6 * nx + 3), es) == 1) return false;
  }
  return true;
}
static_assert(ends(43999999, 1000, 12, 4) && ends(43999999, 1400000, 12, 4) && ends(43997000, 6635, 12, 4), "largest FP32");
static_assert(ends(22300000, 5000, 0, 4) && ends(22300000, 5000, 12, 4) && ends(23400000, 5000, 12, 4), "around 2^31 bytes");
static_assert(ends(43999999, 9000, 0, 2) && ends(43999999, 2900000, 0, 2) && ends(43999999, 43000000, 12, 2), "largest BF16");
static_assert(ends(49, 7, 0, 4) && ends(400, 100, 12, 2), "small");
static_assert(!bf_tap_offset_fits(44000000, 1000, 12, 4) && !bf_tap_offset_fits(43999999, 1500000, 12, 4), "refused");
static_assert(!bf_tap_offset_fits(44000000, 1000, 12, 2) && !bf_tap_offset_fits(1ll << 33, 1 << 16, 12, 2), "refused");
static_assert(!bf_tap_offset_fits(22400000, 5000, 0, 4), "refused from the first plane");
int main() { return 0; }
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_stored_weight_offsets(tmp_path):
    src = tmp_path / "offsets.cpp"
    src.write_text(SOURCE)
    r = subprocess.run(["g++", "-std=c++17", "-fsyntax-only", "-I", CSRC, str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


ORDER = """
#include <cmath>
#include <cstring>
#include "bf_index.h"
long long key(double v) {
  long long b;
  std::memcpy(&b, &v, 8);
  return bf_order_key(b);
}
bool before(double a, int i, double b, int j) { return key(a) < key(b) || (key(a) == key(b) && i < j); }
bool permutation(const double* v, int n) {       // ranks 0 .. n - 1, each taken once
  unsigned seen = 0;
  for (int i = 0; i < n; ++i) {
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += before(v[j], j, v[i], i);
    seen |= 1u << rank;
  }
  return seen == (1u << n) - 1;
}
int main() {
  const double x = std::nan(""), inf = INFINITY;
  const double a[8] = {3, 1, 2, 1, -inf, inf, 0, -0.0}, b[8] = {x, 1, x, 0, 2, x, inf, 1}, c[3] = {x, x, x}, d[2] = {1, x};
  if (!permutation(a, 8) || !permutation(b, 8) || !permutation(c, 3) || !permutation(d, 2)) return 1;
  const double up[] = {-x, -inf, -2, -1, -1e-310, 0, 1e-320, 1, 1.5, 1e300, inf};      // by value
  for (int i = 0; i + 1 < 11; ++i)
    if (!before(up[i], 9, up[i + 1], 1) || before(up[i + 1], 1, up[i], 9)) return 2;
  return key(0.0) == key(-0.0) ? 0 : 3;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_ritz_value_order_is_a_permutation(tmp_path):
    """The Ritz values' ranks index the vectors: they must be a permutation with NaNs among them
    too (places that no rank names would be read uninitialised)."""
    src, exe = tmp_path / "order.cpp", tmp_path / "order"
    src.write_text(ORDER)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True)
    assert subprocess.run([str(exe)]).returncode == 0
