// Eigenbases of the small sectors of classes A-G in one launch (internal).
#pragma once
#include "common.cuh"

namespace caspt2 {

// Largest sector of the one-block solver: two m x m matrices in shared memory.
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
