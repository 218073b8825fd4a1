// Sweep kernels with per-field splitting constants, FP32 bulk (Euler systems only;
// scalar advection has one field).
#include "sweep.cuh"

namespace enoao {

template <int NV, int ORDER>
static const void* field_kernel() {
  return reinterpret_cast<const void*>(sweep_kernel<NV, ORDER, float, false, true>);
}

const void* sweep_fp32_field(int nv, int order) {
  switch (nv * 10 + order) {
    case 35: return field_kernel<3, 5>();
    case 37: return field_kernel<3, 7>();
    case 45: return field_kernel<4, 5>();
    case 47: return field_kernel<4, 7>();
    case 55: return field_kernel<5, 5>();
    case 57: return field_kernel<5, 7>();
    default: return nullptr;
  }
}

}  // namespace enoao
