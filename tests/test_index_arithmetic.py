"""The stored-weight walk's 32-bit byte offsets at the ends of the range it is taken for, in a
constant expression (where a signed overflow does not compile), against 64-bit arithmetic."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1509_02468_gb300", "csrc")

SOURCE = """
#include "bf_index.h"
// first byte of the weight of tap plane f, `shift` samples from pixel i, by both routes
constexpr bool right(long long n, long long i, int f, int shift, int es) {
  const int e = f * (int)n + shift;
  return (unsigned)i * (unsigned)es + bf_byte_offset(e, es) == (unsigned long long)((f * n + i + shift) * es);
}
constexpr long long N = BF_PIPE_W_MAX_N - 1;
static_assert(24 * N * 4 <= 0xffffffffll && 24 * N <= 0x7fffffff, "range of the arithmetic");
static_assert(right(N, N - 1, 23, 0, 4) && right(N, N - 1, 23, -30001, 4) && right(N, N - 1, 0, -30001, 4), "last pixel");
static_assert(right(N, 30001, 0, -30001, 4) && right(N, 0, 23, 0, 4) && right(N, 0, 0, 0, 4), "first pixels");
static_assert(right(N, N / 2, 12, -7, 4) && right(N, N / 2, 13, -7, 2) && right(N, N - 1, 23, -3, 2), "between");
static_assert(right(23400000, 23399999, 23, 0, 4) && right(23300000, 23299999, 23, 0, 4), "either side of 2^31 bytes");
int main() { return 0; }
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_stored_weight_offsets(tmp_path):
    src = tmp_path / "offsets.cpp"
    src.write_text(SOURCE)
    r = subprocess.run(["g++", "-std=c++17", "-fsyntax-only", "-I", CSRC, str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
