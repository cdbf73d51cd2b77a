// Kernels of the bfs child body (see np_bodies.cuh).
#include "np_table.cuh"

namespace nestpar {
const BodyKernels& bfs_kernels() {
  static const BodyKernels t = [] {
    BodyKernels k = with_sweep<BfsSweepBody, 0>(make_table<BfsBody>());
    k.first_levels = (const void*)bfs_first_levels<BfsBody>;
    return k;
  }();
  return t;
}
}  // namespace nestpar
