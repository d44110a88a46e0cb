// Eigenbases of the small sectors of classes A-G in one launch (internal).
#pragma once
#include "common.cuh"

namespace caspt2 {

// Largest sector of the one-block solver.  Two m x m matrices in shared memory would allow 118 rows.
// An eigenproblem takes one block 1.5 ms at 80 rows, 2.0 at 96 and 2.7 at 112, alone on the large
// path 0.75, 0.86 and 1.07; but the sectors of a solve (11, under SS-SR 11 n) run side by side
// here and one after the other there.
constexpr int kSectorBlockMax = 96;

// One sector: class matrices S, F [2][m][m] (identity and pair-swap parts), the sign of the
// swapped part, the selected state (SS-SR; < 0: all), and the outputs Y [msec][nk],
// omega [nk].  X [msec * msec] and scr (sector_block_scratch doubles) are work space.
struct SectorJob {
  const double *S, *F;
  int m, n, Lsel, msec;
  double sgn, thresh;
  double *X, *scr, *Y, *omega;
};
size_t sector_block_scratch(int msec);
// info[2 j] = nk of job j, info[2 j + 1] = -1 when its matrices hold a NaN or an infinity.
cudaError_t sector_block_launch(const SectorJob* jobs, int njobs, int mmax, int* info,
                                cudaStream_t s);

}  // namespace caspt2
