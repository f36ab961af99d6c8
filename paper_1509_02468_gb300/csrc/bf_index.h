// Index arithmetic that host code can check too (no CUDA header needed).
#pragma once

#ifdef __CUDACC__
#define BF_HD __host__ __device__
#else
#define BF_HD
#endif

// Integer that orders doubles (by their bits) as their values do, NaNs before all others: ranks by
// it, ties by place, are a permutation whatever the values are.
BF_HD constexpr long long bf_order_key(long long bits) {
  const long long mag = bits & 0x7fffffffffffffffll;
  return mag > 0x7ff0000000000000ll ? -0x7fffffffffffffffll : (bits < 0 ? -mag : mag);
}

// Byte offsets of the stored-weight walk: 24 planes of n weights of es bytes, rows of nx.  A
// weight is addressed from its pixel's place in plane f0 (unsigned bytes from the first plane on)
// by a signed number of weights, whose product with es stays within an int; the sum is taken
// modulo 2^32.  f0 is the middle plane, 12; counted from the first plane, 0, the product would
// overflow from 2^31 bytes on.  (As unsigned products they make the kernel slower: 2048 x 2048,
// FP32, 16 columns: 385 us against 369.)
BF_HD constexpr unsigned bf_base_offset(unsigned i, unsigned f0, unsigned n, unsigned es) { return (i + f0 * n) * es; }

// e weights from there: (f - f0) planes and what the neighbour is away
BF_HD constexpr unsigned bf_tap_offset(unsigned base, int e, int es) { return base + (unsigned)(e * es); }

// Whether an image may take this arithmetic (shifts reach 3 rows back and, in a strip's rows
// past the image, 6 on; pixel numbers in the last tiles go 48 rows past it).
constexpr int BF_PIPE_W_MAX_N = 44000000;
BF_HD constexpr bool bf_tap_offset_fits(long long n, long long nx, int f0, int es) {
  return n < BF_PIPE_W_MAX_N && 24 * n * es < (1ll << 32) && n + 48 * nx < (1ll << 31) &&
         ((f0 > 12 ? f0 : 24 - f0) * n + 6 * nx + 3) * es < (1ll << 31);
}
