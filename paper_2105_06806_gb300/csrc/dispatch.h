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

// Sector-order FP32 product through block-major order (two permutations and
// the orbital-factorised product in a scratch pair of vectors) instead of the
// sector-order kernel, whose H_up hops gather across whole CSR rows and cost
// the more the longer those are (D_up).  Sector-order kernel / detour, measured
// on 230 sectors of Ns=14-20, with and without exchange terms:
//   two, three orbitals: D_up from 8008 on 1.06 to 1.9 (Norb=2 Ns=16 (8,8) 2724
//     / 1950 us; 2.1 to 4.0 with two down electrons), with fewer than 5 * 2^20
//     elements only from 11440 on (8008: 0.93); 5005 and 6435 from 5 * 2^20
//     elements on 1.0 to 1.43, below that down to 0.83; up to 3432 0.85 to 1.24
//     either way (Norb=2 Ns=14 (7,7) 146 / 158 us, Norb=3 Ns=15 (5,7) 257 / 269);
//   four orbitals: D_up from 12870 on 1.01 to 3.6, 11440 from 2^25 elements on
//     1.01 to 1.1, below that and with shorter rows 0.70 to 0.99;
//   five orbitals: 0.59 to 0.84 without exchange terms, 0.86 to 1.2 with them.
// group: levels of an orbital group, 0 where the factorised product does not
// apply; pinned: the kernel the caller chose for the block-major layout (0 the
// tiled family, which is then taken from 2^20 elements on, 1 element-parallel,
// -1 none).  The scratch stays cached in the library's pool, so it is bounded:
// above ED_PERMUTE_SCRATCH_MAX the sector-order kernel runs.
constexpr int64_t ED_PERMUTE_MIN = (int64_t)1 << 20;
constexpr int64_t ED_PERMUTE_SCRATCH_MAX = (int64_t)2 << 30;
constexpr int64_t ed_permute_scratch(int64_t bdim) { return 2 * bdim * (int64_t)sizeof(float); }
constexpr bool ed_takes_permuted(int norb, int group, int64_t dup, int64_t dim, int64_t bdim,
                                 int pinned) {
  if (group == 0 || dim < ED_PERMUTE_MIN || pinned == 1 ||
      ed_permute_scratch(bdim) > ED_PERMUTE_SCRATCH_MAX)
    return false;
  if (pinned == 0) return true;
  if (norb <= 3) return dup >= (dim >= (int64_t)5 << 20 ? 5000 : 11000);
  return norb == 4 && dup >= (dim >= (int64_t)1 << 25 ? 11000 : 12000);
}

// Size class of the autotuner's key.  Sectors of at most 2^17 padded elements
// are not timed.  In FP32 the faster kernel of a model shape changes with the
// size (element-parallel / tiled ms: Norb=2 Ns=14 0.5 at 1e6 elements, 1.3 at
// 1.2e7; Norb=3 0.25 at Ns=12, 2.3 at Ns=18), so there are three classes: over
// 457 sectors of 15 shapes within three electrons of half filling, the choice
// of a class's first sector costs the others 2.2% on average (3.6% with one
// class per shape, up to 3.1 times; 1.9% with a class per factor of 8, whose
// boundaries run between the half-filled sector of an odd Ns and its
// neighbours: a solve would time both).  In FP64 the element-parallel kernel was
// the faster one throughout: one class, no further timing.
constexpr int64_t ED_TUNE_MIN = (int64_t)1 << 17;
constexpr int ed_tune_class(int elem, int64_t bdim) {
  return elem != 4 ? 0 : (bdim >= (int64_t)1 << 20) + (bdim >= (int64_t)13 << 20);
}
