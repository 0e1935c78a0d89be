// stage_cols_f32.cu -- column passes of the transport stages in single precision.
#include "stage_launch.cuh"

namespace reg {
namespace fused {
REG_COLS_OF(float)
}  // namespace fused
}  // namespace reg
