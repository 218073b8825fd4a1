// FP32-bulk sweep kernels of ENO-AO7 (state and Runge-Kutta combine in FP64)
// that re-decide their near-ties in the sweep, and their TMA-staged variant.
#include "sweep_shapes.cuh"

namespace enoao {

template <int NV>
static const void* tma_kernel() {
  return reinterpret_cast<const void*>(sweep_kernel<NV, 7, float, false, false, true>);
}

const void* sweep_fp32_o7(int nv, int shape, int variant) {
  if (variant != kSweepFp32Tma) return kernel_by_shape<7, float>(nv, shape);
  switch (nv) {
    case 1: return tma_kernel<1>();
    case 3: return tma_kernel<3>();
    case 4: return tma_kernel<4>();
    case 5: return tma_kernel<5>();
    default: return nullptr;
  }
}

}  // namespace enoao
