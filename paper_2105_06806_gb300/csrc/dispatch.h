// Rules of the product dispatch that need no device: plain host code, so that
// they can be checked at sizes no test allocates.
#pragma once

#include <stdint.h>

// Element-parallel product: rows per thread of k_hv_rows.
constexpr int HVS_ROWS = 4;

// Work units of k_hv_rows: (group of HVS_ROWS rows, padded column).
constexpr int64_t ed_rows_units(int64_t ddw, int64_t stride) {
  return (ddw + HVS_ROWS - 1) / HVS_ROWS * stride;
}

// True where the element-parallel product takes k_hv_rows: in FP32 above 2^22
// elements a thread takes one column of 4 consecutive rows, which share the
// column's tables and H_up entries and have their gathers in flight together
// (Norb=5 Ns=15 509 -> 367 us, Norb=1 Ns=15 491 -> 411 us).  Smaller sectors
// need the threads (1-2% slower at 10^6 elements), and FP64 is bound by its
// pipe (5.80 against 5.57 ms at Norb=2 Ns=16).  The kernel finds its row with a
// 32-bit division, so above 2^32 units (FP32 vectors of 69 GB) k_hv_small,
// which indexes in 64 bits, keeps the work.
constexpr bool ed_takes_rows(int elem, int64_t ddw, int64_t stride) {
  return elem == 4 && ddw * stride > (int64_t)1 << 22 &&
         ed_rows_units(ddw, stride) <= (int64_t)1 << 32;
}
