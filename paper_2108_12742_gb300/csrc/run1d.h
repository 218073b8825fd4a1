// The persistent run of small 1D problems (run1d.cu).
#pragma once

#include <cuda_runtime.h>

#include "enoao_internal.h"
#include "step_state.cuh"

namespace enoao {

struct Run1dArgs {
  SweepArgs stage[3];  // the sweeps of the three Runge-Kutta stages
  StepConsts k;
  long long cap;       // steps of this launch at most
  unsigned polls;      // bound on a block's polls of the grid barrier
};

constexpr int kRun1dMaxTile = 256;
constexpr unsigned kRun1dPolls = 1u << 22;  // a few seconds

// Cells per tile and threads per block for a problem of n cells.
void run1d_tile(int nv, long long n, int sms, int* ts, int* block);
// fp32: bulk precision.  One cooperative launch, a block per tile;
// cudaErrorCooperativeLaunchTooLarge (and nothing launched) where the blocks
// cannot all be resident at once, or are more than max_blocks (if that is >= 0).
cudaError_t run1d_launch(int nv, int order, int fp32, const Run1dArgs& a, int block, int sms,
                         int max_blocks, cudaStream_t s);

}  // namespace enoao
