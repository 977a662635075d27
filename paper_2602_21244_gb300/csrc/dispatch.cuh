// Rules that choose between kernels by the sizes of a call.  Plain C++: times
// in us on GB300 (152 SMs); sizes per SM so that the rules scale with the chip.
#pragma once
#include <stdint.h>

namespace dsmc {

// Cell moments and moment matching (match): claims of cells by warps that stay
// (k_cells), or one group of cells per warp with 8 or 32 lanes per cell
// (k_cells_once).  Direct calls, by claims / by groups:
//   20 particles a cell   match 12 / 9 at 1,000 cells, 22 / 17 at 10,000, 25 / 22 at 19,456, 30 / 32 at 30,000,
//                         moments 16 / 11 at 14,400, 21.0 / 19.5 at 40,000, 23.0 / 22.9 at 48,640
//   61 on average, up to  match 33 / 27 at 6,000 cells, 37 / 36 at 9,375, 37 / 41 at 13,500, 40 / 52 at 18,375,
//   250 (dense cells      moments 23 / 16 at 6,000, 30 / 26 at 18,375, 33 / 35 at 30,375, 39 / 43 at 45,375
//   side by side)
// The groups save the claims' chain but pay the FP64 remainder per group of 4
// cells instead of per 16, and in matching a dense cell holds up its group: so
// the limits lie by cells, for matching lower where the number of particles is
// not known (n = 0: a direct call, the cell starts are in device memory), and
// by particles where it is (a step).  Up to 8 cells per SM 32 lanes per cell,
// however many particles (1,000 cells of 200: match 12 by 32 lanes, 20 by 8, 28 by
// claims; of 1,000: 31, 103, 98).
enum CellKernel { CELLS_CLAIMED = 0, CELLS_ONCE_8 = 8, CELLS_ONCE_32 = 32 };
constexpr int64_t kByClaims = -1;   // in the place of n: k_cells, the kernel that the tuned shapes are for

// Cells that k_cells gives to a block at least.
constexpr int kCellsPerBlock = 32;

inline CellKernel cells_kernel(bool match, int64_t n_cells, int64_t n, int64_t sms) {
  if (n == kByClaims) return CELLS_CLAIMED;
  if (n_cells <= 8 * sms) return CELLS_ONCE_32;
  if (n_cells > (!match ? 320 : n > 0 ? 128 : 96) * sms || n > (match ? 2500 : 10000) * sms) return CELLS_CLAIMED;
  return CELLS_ONCE_8;
}

// The pair update of a step on the VHS (table false) and look-up paths: by
// groups of cells (k_collide_groups, one warp per group), or by stamps
// (k_collide_vhs, k_collide_table, every SM on every cell's pairs).  Whole
// step, by stamps / by groups, pairs a particle in brackets:
//   VHS       1,024 cells of 60 [0.6] 120 / 96, of 400 269 / 255, of 1,000 540 / 528; 6,000 of 60 177 / 164, of 120
//             221 / 246; 9,700 of 20 159 / 148, of 60 [0.15] 159 / 151, [0.6] 210 / 211, of 120 268 / 311
//   look-up   1,024 cells of 60 [0.8] 137 / 101, of 400 393 / 343; 9,000 of 60 250 / 216; 30,000 of 20 281 / 243, of
//             60 394 / 457, of 120 637 / 807; 43,000 of 20 325 / 305; of the hypersonic gas (61 a cell, up to
//             250) 37,500 638 / 569, 73,500 926 / 926
//   few cells, very dense: 16 cells of 400 [0.6] VHS 137 / 130, of 1,000 264 / 278, of 4,000 1536 / 1585; look-up
//             220 / 214, 540 / 564, 3182 / 3305; 64 of 4,000 1587 / 1634, 3309 / 3418; one of 4,000 [1.3] VHS 603 / 781
// Groups save the stamps and the waits between a cell's rounds; larger gases
// fill the chip without that, and a very dense cell is one warp's work.
inline bool groups_suit(bool table, int64_t n_cells, int64_t n, int64_t sms) {
  return n_cells <= (table ? 288 : 64) * sms && n <= (table ? 16000 : 4000) * sms && n <= 512 * n_cells;
}

}  // namespace dsmc
