// FP64 sweep kernels (every step of the path in double precision).
#include "sweep_shapes.cuh"

namespace enoao {

const void* sweep_fp64(int nv, int order, int shape) {
  return order == 5 ? kernel_by_shape<5, double>(nv, shape)
                    : (order == 7 ? kernel_by_shape<7, double>(nv, shape) : nullptr);
}

}  // namespace enoao
