// Launchers of the float32 strided-axis kernels (all supported y and z extents).
#include "launch.cuh"
namespace cbs {
CBS_ROW_LAUNCHERS(extern template, float)
CBS_AXIS_LAUNCHERS(template, float)
}
