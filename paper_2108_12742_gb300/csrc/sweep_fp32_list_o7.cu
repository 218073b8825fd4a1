// FP32-bulk sweep kernels of ENO-AO7 that list their near-ties for the
// grid-wide re-decision pass.
#include "sweep_shapes.cuh"

namespace enoao {

const void* sweep_fp32_list_o7(int nv, int shape) {
  return kernel_by_shape<7, float, true>(nv, shape);
}

}  // namespace enoao
