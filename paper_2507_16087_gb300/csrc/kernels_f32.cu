// Launchers of the float32 row kernels (all supported x extents).
#include "launch.cuh"
namespace cbs {
CBS_AXIS_LAUNCHERS(extern template, float)
CBS_ROW_LAUNCHERS(template, float)
}
