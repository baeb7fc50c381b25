// Column work lists of 3D plans: the prepared tap rows of the column spread (columns.cu).
//
// A column is a kColX x kColY block of fine cells in x-y with all its z-planes.  A node visits
// every column its w x w footprint reaches; a column's visits are sorted by first z tap and z
// class (nodes with the same psi_z row, e.g. one quadrature ring).  Groups of at most 32 visits
// and 8 runs (a run: consecutive visits of one z class) are what a warp takes at a time; what
// it needs of them does not change between evaluations, so the plan stores it ready to use:
// per group one contiguous image
//   X rows   [8 / EPC][32] 16-byte chunks: psi_x of each visit at the column's 8 x cells, zero
//            outside the footprint (read by a lane per visit: conflict-free 16-byte loads)
//   Y rows   [8][32]: the same along y, one row per y cell, so that a lane that holds a cell
//            reads the factors of two consecutive visits in one load; runs start at even visits
//            (an odd run ends with an empty visit) and the row stride spreads the rows over the
//            banks
//   Z rows   [8 runs]: the run's psi_z, tap k at index (first tap + k) mod w, the register that
//            holds that plane
//   head     [8 runs]: first z tap << 12 | end visit << 6 | first visit; visits; runs
#pragma once
#include "common.cuh"

namespace ddi {

template <typename T, int W>
struct ColImage {
  static constexpr int EPC = 16 / (int)sizeof(T);    // values per 16-byte chunk
  static constexpr int CH = 8 / EPC;                  // chunks per X row of 8 values
  static constexpr int RS = 32 * (int)sizeof(T) + 16; // bytes between Y rows
  static constexpr int ZS = (W * (int)sizeof(T) + 15) / 16 * 16;
  static constexpr int X = 0, Y = CH * 512, Z = Y + 8 * RS, HEAD = Z + kColRuns * ZS;
  static constexpr int COUNTS = HEAD + kColRuns * 4;  // int visits (empty ones included), int runs
  static constexpr int BYTES = (COUNTS + 8 + 15) / 16 * 16;
};

// 2D: blocks of kColX x kColY cells; a group is 32 visits of one block and its image the X rows and
// Y rows alone.
template <typename T>
struct BlockImage {
  static constexpr int EPC = 16 / (int)sizeof(T);
  static constexpr int CH = 8 / EPC;
  static constexpr int RS = 32 * (int)sizeof(T) + 16;
  static constexpr int X = 0, Y = CH * 512;
  static constexpr int BYTES = Y + 8 * RS;
};

}  // namespace ddi
