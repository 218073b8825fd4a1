// Whole runs of small 1D problems in one persistent launch: each block owns a
// tile of the grid and takes it through every stage of every step; the blocks
// meet at a grid barrier after each stage and after the step's bookkeeping.
//
// What bounds such a run is latency, not work: a stage of 2000 cells is a few
// microseconds of dependent FP64 operations.  As one graph node per stage it
// also paid for a launch, the sweep's prologue and a bookkeeping node (39 us a
// step at N = 2000, FP64), and steps came in multiples of 32 to 128.  Here a
// tile per SM spreads the cells thinnest, the barrier is one atomic and one
// poll, and the launch ends with the run.  Advection N = 200 to t = 2 (401
// steps) 9.0 -> 5.2 ms, Euler N = 2000 over 120 steps 10.0 -> 5.8 ms.
//
// Every block is resident (a cooperative launch of at most a block per SM), so
// the barrier cannot wait for a block that has not started; its polls are
// bounded all the same: a block that gives up sets the error word and leaves.
// The others then run out of polls at the next barrier, which it never reaches.
// The barrier's count is left short: until the state is set anew (which clears
// it) a launch finds the error word and leaves at once.
#include <algorithm>

#include "run1d.h"
#include "sweep.cuh"

namespace enoao {

namespace {

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// All threads of all blocks; false when the wait ran out.  What a block wrote
// before it (any thread) is seen by every block's L2 reads after it.
__device__ __forceinline__ bool grid_barrier(StepState* st, unsigned limit) {
  __shared__ bool s_ok;
  __syncthreads();
  if (gridDim.x == 1) {
    if (threadIdx.x == 0) __threadfence();  // thread 0 reads what others' atomics left
    return true;
  }
  if (threadIdx.x == 0) {
    bool ok = true;
    __threadfence();
    const unsigned gen = load_acquire(&st->grid_gen);
    if (atomicAdd(&st->grid_count, 1u) == gridDim.x - 1) {
      st->grid_count = 0u;
      __threadfence();
      atomicAdd(&st->grid_gen, 1u);
    } else {
      unsigned polls = 0;
      while (load_acquire(&st->grid_gen) == gen && ok) ok = polls++ < limit;
      if (!ok) atomicOr(&st->err, kErrBarrier);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok;
}

template <int NV, int ORDER, typename R>
__global__ void __launch_bounds__(256, 1) run1d_kernel(const __grid_constant__ Run1dArgs P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ TileConst<R> s_k;
  __shared__ TileGeo s_geo;
  __shared__ int s_skip, s_par;
  __shared__ double s_red[8];
  StepState* st = P.stage[0].st;
  unsigned long long nfall = 0;
  if (threadIdx.x == 0) {
    s_geo = tile_geo(P.stage[0], blockIdx.x);
    s_skip = __ldcg(&st->err) & kErrBarrier;
  }
  __syncthreads();
  if (s_skip) return;
  bool ok = true;
  long long n = 0;
  for (; n < P.cap; ++n) {
    if (blockIdx.x == 0 && threadIdx.x == 0) begin_step(st, P.k);
    ok = grid_barrier(st, P.polls);
    if (!ok) break;
    if (threadIdx.x == 0) {
      s_skip = __ldcg(&st->skip);
      s_par = __ldcg(&st->par);
    }
    __syncthreads();
    if (s_skip) break;
    double amax[3] = {0.0, 0.0, 0.0};
    for (int stage = 0; stage < 3 && ok; ++stage) {
      const SweepArgs& A = P.stage[stage];
      if (threadIdx.x == 0)
        tile_const<ORDER, R>(A, __ldcg(&st->alpha[0]), __ldcg(&st->dt), s_k);
      __syncthreads();
      sweep_tile<NV, ORDER, R, true, false, false, false, kShapeXCombine>(A, s_geo, smem_raw, s_k,
                                                                          amax, nfall);
      if (NV > 1 && stage == 2) {
        double v = amax[0];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
        if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
          for (int w = 1; w < (int)blockDim.x >> 5; ++w) v = fmax(v, s_red[w]);
          if (v > 0.0)
            atomicMax(&st->alpha_acc[s_par][0], (unsigned long long)__double_as_longlong(v));
        }
      }
      ok = grid_barrier(st, P.polls);
    }
    if (!ok) break;
  }
  if (sizeof(R) == 4 && nfall) atomicAdd(&st->fallbacks, nfall);
  // every block is past the last stage's barrier
  if (ok && n == P.cap && blockIdx.x == 0 && threadIdx.x == 0) finalize_pending(st);
}

template <int NV, int ORDER, typename R>
cudaError_t launch_one(const Run1dArgs& a, int block, int sms, int max_blocks, cudaStream_t s) {
  const SweepArgs& A = a.stage[0];
  const size_t smem = sweep_smem_bytes(NV, sizeof(R) == 4, 1, A.se);
  const void* kernel = reinterpret_cast<const void*>(run1d_kernel<NV, ORDER, R>);
  int per_sm = 0;
  cudaError_t e = sweep_setup(kernel, block, smem, &per_sm);
  if (e != cudaSuccess) return e;
  if (A.ntiles > (long long)per_sm * sms || (max_blocks >= 0 && A.ntiles > max_blocks))
    return cudaErrorCooperativeLaunchTooLarge;
  void* args[1] = {const_cast<Run1dArgs*>(&a)};
  return cudaLaunchCooperativeKernel(kernel, dim3((unsigned)A.ntiles), dim3(block), args, smem, s);
}

}  // namespace

// Scalar problems whose extended cells fit one block's threads once stay in one
// block: a stage is less than a grid barrier there (N = 200: 13.3 us a step, 15.3
// in tiles of 63; N = 400: 19.0 in one block, 14.7 in tiles of 63, 18.5 of 15).
// The Euler equations take a tile per SM, of at least 15 cells (16 faces: the
// face groups of a tile fill one round of 128 threads).
void run1d_tile(int nv, long long n, int sms, int* ts, int* block) {
  const long long per_sm = (n + sms - 1) / sms;
  long long t = nv == 1 ? (n <= 246 ? n : std::max<long long>(63, per_sm))
                        : std::max<long long>(15, per_sm);
  *ts = (int)t;
  *block = t > 120 ? 256 : 128;
}

cudaError_t run1d_launch(int nv, int order, int fp32, const Run1dArgs& a, int block, int sms,
                         int max_blocks, cudaStream_t s) {
  switch (nv * 100 + order * 10 + (fp32 ? 1 : 0)) {
    case 150: return launch_one<1, 5, double>(a, block, sms, max_blocks, s);
    case 170: return launch_one<1, 7, double>(a, block, sms, max_blocks, s);
    case 151: return launch_one<1, 5, float>(a, block, sms, max_blocks, s);
    case 171: return launch_one<1, 7, float>(a, block, sms, max_blocks, s);
    case 350: return launch_one<3, 5, double>(a, block, sms, max_blocks, s);
    case 370: return launch_one<3, 7, double>(a, block, sms, max_blocks, s);
    case 351: return launch_one<3, 5, float>(a, block, sms, max_blocks, s);
    case 371: return launch_one<3, 7, float>(a, block, sms, max_blocks, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace enoao
