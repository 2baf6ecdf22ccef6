// Instantiations of the float step kernel on opposite pairs: 2-D shapes.
#include "rt_shapes.h"
#include "rt_step_sym.cuh"

namespace rtg {

cudaError_t launch_s2(const StepArgs<float> &a, const stepk::SymTable &tab, bool vel, TileShape t, cudaStream_t s) {
#define RT_CASE(X, Y, Z)                                                          \
  if (t.tx == X && t.ty == Y && t.tz == Z)                                        \
    return vel ? stepk::launch_shape_sym<2, true, X, Y, Z>(a, tab, s)             \
               : stepk::launch_shape_sym<2, false, X, Y, Z>(a, tab, s);
  RT_SHAPES_F2(RT_CASE)
#undef RT_CASE
  return cudaErrorInvalidConfiguration;
}

}  // namespace rtg
