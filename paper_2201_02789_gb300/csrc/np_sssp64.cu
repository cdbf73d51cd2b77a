// Kernels of the packed-distance SSSP child body (see np_bodies.cuh).
#include "np_table.cuh"

namespace nestpar {
const BodyKernels& sssp64_kernels() {
  static const BodyKernels t = [] {
    BodyKernels k = with_sweep<Sssp64SweepBody, 1>(make_table<Sssp64Body>());
    k.level_small = (const void*)sssp_cluster<Sssp64Body>;
    k.level_small_smem = (int)kClusterSmem;
    k.level_small_cluster = true;
    return k;
  }();
  return t;
}
}  // namespace nestpar
