// Launchers of the float64 row kernels (all supported x extents).
#include "launch.cuh"
namespace cbs {
CBS_AXIS_LAUNCHERS(extern template, double)
CBS_ROW_LAUNCHERS(template, double)
}
