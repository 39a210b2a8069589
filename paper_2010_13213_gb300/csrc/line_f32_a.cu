// Line transforms of 16 points per second step, NB = 1..6, and of 8 points, NB = 2 and 4, arithmetic float.
#include "line_ops.cuh"

namespace lgf {
LINE_RANGE_DEFINE(float, 16, 1, 6, 1)
LINE_RANGE_DEFINE(float, 8, 2, 4, 2)
}  // namespace lgf
