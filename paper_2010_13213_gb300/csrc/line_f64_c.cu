// Line transforms of 16 points per second step, NB = 12..16, arithmetic double.
#include "line_ops.cuh"

namespace lgf {
LINE_RANGE_DEFINE(double, 16, 12, 16, 1)
}  // namespace lgf
