// Index arithmetic that host code can check too (no CUDA header needed).
#pragma once

#ifdef __CUDACC__
#define BF_HD __host__ __device__
#else
#define BF_HD
#endif

// Byte offset of element e (of es bytes; negative: before) as an unsigned number, to be added to a
// pixel's unsigned byte offset: the sum is taken modulo 2^32 and is right wherever the element
// lies in the first 2^32 bytes.  (As signed numbers the product overflows from 2^31 bytes on.)
BF_HD constexpr unsigned bf_byte_offset(int e, int es) { return (unsigned)e * (unsigned)es; }

// Samples below which the stored-weight walk may take this arithmetic: its 24 planes of at most
// four bytes lie below 2^32 bytes, its element numbers below 2^31.
constexpr int BF_PIPE_W_MAX_N = 44000000;
