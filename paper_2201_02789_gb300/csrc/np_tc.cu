// Kernels of the triangle-counting child body (see np_bodies.cuh).
#include "np_table.cuh"
#include "np_tc.cuh"

namespace nestpar {
const BodyKernels& tc_kernels() {
  static const BodyKernels t = [] {
    BodyKernels k = make_table<TcBody>();
    k.map_child = (const void*)tc_child;
    k.map_vertices = kTcMaxVertices;
    return k;
  }();
  return t;
}
}  // namespace nestpar
