// Launchers of the float64 strided-axis kernels (all supported y and z extents).
#include "launch.cuh"
namespace cbs {
CBS_ROW_LAUNCHERS(extern template, double)
CBS_AXIS_LAUNCHERS(template, double)
}
