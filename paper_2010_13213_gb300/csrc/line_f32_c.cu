// Line transforms of 16 points per second step, NB = 12..16, arithmetic float.
#include "line_ops.cuh"

namespace lgf {
LINE_RANGE_DEFINE(float, 16, 12, 16, 1)
}  // namespace lgf
