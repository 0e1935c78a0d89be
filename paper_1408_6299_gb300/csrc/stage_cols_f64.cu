// stage_cols_f64.cu -- column passes of the transport stages in double precision.
#include "stage_launch.cuh"

namespace reg {
namespace fused {
REG_COLS_OF(double)
}  // namespace fused
}  // namespace reg
