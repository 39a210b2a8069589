// Line transforms of 8 points per second step, NB = 1..15, arithmetic double.
#include "line_ops.cuh"

namespace lgf {
LINE_RANGE_DEFINE(double, 8, 1, 15, 2)
}  // namespace lgf
