// The fused 2D stage kernel (both axes of one Runge-Kutta stage in one
// launch), FP32 bulk, for the 2D systems (scalar advection and Euler).
#include "sweep.cuh"

namespace enoao {

template <int NV, int ORDER>
static const void* fused_kernel() {
  return reinterpret_cast<const void*>(fused2d_kernel<NV, ORDER>);
}

const void* fused2d_kernel_for(int nv, int order) {
  switch (nv * 10 + order) {
    case 15: return fused_kernel<1, 5>();
    case 17: return fused_kernel<1, 7>();
    case 45: return fused_kernel<4, 5>();
    case 47: return fused_kernel<4, 7>();
    default: return nullptr;
  }
}

}  // namespace enoao
