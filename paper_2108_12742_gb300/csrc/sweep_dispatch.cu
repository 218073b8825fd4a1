// The sweep kernel of a launch, and the launches of the grid-wide re-decision
// pass.
#include "sweep.cuh"

namespace enoao {

const void* sweep_kernel_for(int nv, int order, int shape, int variant) {
  const bool o5 = order == 5;
  if (!o5 && order != 7) return nullptr;
  switch (variant) {
    case kSweepFp32:
    case kSweepFp32Tma:
      return o5 ? sweep_fp32_o5(nv, shape, variant) : sweep_fp32_o7(nv, shape, variant);
    case kSweepFp32List:
      return o5 ? sweep_fp32_list_o5(nv, shape) : sweep_fp32_list_o7(nv, shape);
    case kSweepFp64: return sweep_fp64(nv, order, shape);
    case kSweepFp32Field: return sweep_fp32_field(nv, order);
    case kSweepFp64Field: return sweep_fp64_field(nv, order);
    default: return nullptr;
  }
}

template <int NV, int ORDER>
static cudaError_t redo_one(const SweepArgs& a, int grid, cudaStream_t s) {
  redo_kernel<NV, ORDER><<<grid, 128, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  redo_apply_kernel<NV><<<grid, 128, 0, s>>>(a);
  return cudaGetLastError();
}

// The grid-wide FP64 re-decision pass of a sweep launched with a.redo set (two
// kernels, stream-ordered after the sweep).
cudaError_t redo_launch_fp32(int nv, int order, const SweepArgs& a, int grid, cudaStream_t s) {
  switch (nv * 10 + order) {
    case 15: return redo_one<1, 5>(a, grid, s);
    case 17: return redo_one<1, 7>(a, grid, s);
    case 35: return redo_one<3, 5>(a, grid, s);
    case 37: return redo_one<3, 7>(a, grid, s);
    case 45: return redo_one<4, 5>(a, grid, s);
    case 47: return redo_one<4, 7>(a, grid, s);
    case 55: return redo_one<5, 5>(a, grid, s);
    case 57: return redo_one<5, 7>(a, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace enoao
