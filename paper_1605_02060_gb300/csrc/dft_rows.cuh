// Where the rows of a real-DFT table lie.  Plain C++ apart from the execution space, so that the
// offsets of long axes can be checked on the host.
#pragma once

#ifdef __CUDACC__
#define LDDMM_ROWS __host__ __device__ __forceinline__
#else
#define LDDMM_ROWS inline
#endif

namespace lddmm {

// Row of the cosine of frequency p (row 0: the constant); the sine's row is 2 p.
LDDMM_ROWS int fold_row_c(int p) { return p ? 2 * p - 1 : 0; }

// Bytes from the start of a float table [n][n] to that row, n4 = 4 n.  64 bits, from a 32-bit
// product (one instruction with the address it is added to): the table of an axis past 46340 has
// more than 2^31 elements, while the field's own offsets stay below.
LDDMM_ROWS unsigned long long fold_row_bytes(int p, unsigned n4) {
  return (unsigned long long)(unsigned)fold_row_c(p) * n4;
}

}  // namespace lddmm
