// Line transforms of 16 points per second step, NB = 7..11, arithmetic df.
#include "line_ops.cuh"

namespace lgf {
LINE_RANGE_DEFINE(df, 16, 7, 11, 1)
}  // namespace lgf
