// FP32-bulk sweep kernels of ENO-AO5 that list their near-ties for the
// grid-wide re-decision pass.
#include "sweep_shapes.cuh"

namespace enoao {

const void* sweep_fp32_list_o5(int nv, int shape) {
  return kernel_by_shape<5, float, true>(nv, shape);
}

}  // namespace enoao
