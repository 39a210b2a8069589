// Line transforms of 16 points per second step, NB = 12..16, arithmetic df.
#include "line_ops.cuh"

namespace lgf {
LINE_RANGE_DEFINE(df, 16, 12, 16, 1)
}  // namespace lgf
