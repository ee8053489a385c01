// Sizes of the banded preconditioner's solves (k_band.cu): the same functions for the
// planner, the launch and the kernel, and on the CPU alone for their tests.
#ifndef FOCK_BAND_PLAN_H
#define FOCK_BAND_PLAN_H

#include <stddef.h>

#ifdef __CUDACC__
#define FOCK_HD __host__ __device__
#else
#define FOCK_HD
#endif

namespace fock {

// A banded factor is made up to this many operations.
constexpr double kBandFlops = 8e9;
inline bool band_rule(int L, int D, int m0) {
  return 2.0 * L * (double)D * D * (double)m0 * m0 * m0 <= kBandFlops;
}

// doubles of one step of the banded solves with nd block coefficients, padded to 16 bytes
FOCK_HD inline size_t band_step(int nd, int m0) { return ((size_t)nd * m0 * m0 + 1) & ~(size_t)1; }

constexpr int kBandStage = 8192;   // doubles of a stage of coefficients that every launch can hold twice

// Coefficient rows per stage of `stage` doubles: the whole step, else a multiple of 8, else an
// even number (a piece then starts on a 16-byte boundary).  Up to kBandFlops a row takes at
// most 1620 doubles, so two always fit.
FOCK_HD inline int band_rows(int nd, int m0, int stage) {
  if ((int)band_step(nd, m0) <= stage) return m0;
  const int r = stage / (nd * m0);
  return r >= 8 ? r & ~7 : r & ~1;
}
// doubles of piece h of a step of `total` doubles, `rows` rows of `width` a piece
FOCK_HD inline int band_piece(int rows, int width, int total, int h) {
  const int left = total - h * rows * width;
  return rows * width < left ? rows * width : left;
}

// The stage that a task would have: eight rows, of blocks up to 8 functions the whole step.
inline int band_stage_rows8(int D, int m0) { return m0 > 8 ? 8 * (D + 1) * m0 : (int)band_step(D + 1, m0); }
// rows of the ring, of z and of the middle that a column keeps beside the two stages
inline int band_side_rows(int D, int m0, bool twist) { return ((twist ? 3 : 1) * D + 4) * m0; }

// Doubles of a stage for tasks whose largest step, band_stage_rows8 and band_side_rows these
// are, with `room` doubles of shared memory: a whole step up to 64 KB or eight rows, where that
// fits beside the rows (a task alone always does), else 64 KB, whatever number of rows that is.
inline int band_stage(int maxstep, int max8, int maxrow, int room) {
  const int least = maxstep < kBandStage ? maxstep : kBandStage, s = max8 > least ? max8 : least;
  return 2 * (long long)s + maxrow <= room ? s : least;
}

}  // namespace fock

#endif
