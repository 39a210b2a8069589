// Line transforms of 16 points per second step, NB = 7..11, arithmetic float.
#include "line_ops.cuh"

namespace lgf {
LINE_RANGE_DEFINE(float, 16, 7, 11, 1)
}  // namespace lgf
