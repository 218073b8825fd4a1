// Kernel tables of the instantiation units: the sweep kernel of one precision,
// order and variant by system and shape (only the shapes a system meets).
#pragma once

#include "sweep.cuh"

namespace enoao {

template <int NV, int ORDER, typename R, bool DEFER, int SHAPE>
const void* shape_kernel() {
  return reinterpret_cast<const void*>(sweep_kernel<NV, ORDER, R, DEFER, false, false, SHAPE>);
}

// 1D combines along x; 2D stores x and combines y; 3D stores x and y and
// combines z.  The listing variant (DEFER) never writes fluxes.
template <int ORDER, typename R, bool DEFER = false>
const void* kernel_by_shape(int nv, int shape) {
  switch (nv * 10 + shape) {
    case 10 + kShapeXStore: return shape_kernel<1, ORDER, R, DEFER, kShapeXStore>();
    case 10 + kShapeXCombine: return shape_kernel<1, ORDER, R, DEFER, kShapeXCombine>();
    case 10 + kShapeYStore: return shape_kernel<1, ORDER, R, DEFER, kShapeYStore>();
    case 10 + kShapeYCombine: return shape_kernel<1, ORDER, R, DEFER, kShapeYCombine>();
    case 30 + kShapeXCombine: return shape_kernel<3, ORDER, R, DEFER, kShapeXCombine>();
    case 40 + kShapeXStore: return shape_kernel<4, ORDER, R, DEFER, kShapeXStore>();
    case 40 + kShapeYCombine: return shape_kernel<4, ORDER, R, DEFER, kShapeYCombine>();
    case 50 + kShapeXStore: return shape_kernel<5, ORDER, R, DEFER, kShapeXStore>();
    case 50 + kShapeYStore: return shape_kernel<5, ORDER, R, DEFER, kShapeYStore>();
    case 50 + kShapeYCombine: return shape_kernel<5, ORDER, R, DEFER, kShapeYCombine>();
    default: break;
  }
  if constexpr (!DEFER) {
    switch (nv * 10 + shape) {
      case 10 + kShapeFlux: return shape_kernel<1, ORDER, R, false, kShapeFlux>();
      case 30 + kShapeFlux: return shape_kernel<3, ORDER, R, false, kShapeFlux>();
      case 40 + kShapeFlux: return shape_kernel<4, ORDER, R, false, kShapeFlux>();
      case 50 + kShapeFlux: return shape_kernel<5, ORDER, R, false, kShapeFlux>();
      default: break;
    }
  }
  return nullptr;
}

}  // namespace enoao
