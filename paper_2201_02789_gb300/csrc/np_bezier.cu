// Kernels of the bezier child body (see np_bodies.cuh).
#include "np_points.cuh"
#include "np_table.cuh"

namespace nestpar {
const BodyKernels& bezier_kernels() {
  static const BodyKernels t = [] {
    BodyKernels k = make_table<BezierBody>();
    k.points_count = (const void*)bezier_count;
    k.points = (const void*)bezier_points;
    k.points_fused = (const void*)bezier_fused;
    return k;
  }();
  return t;
}
}  // namespace nestpar
