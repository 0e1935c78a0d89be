// stage_rows_f32.cu -- advection row passes of the transport stages in single precision.
#include "stage_launch.cuh"

namespace reg {
namespace fused {
REG_ROWS_OF(float, EPI_ADV2)
REG_ROWS_OF(float, EPI_ADV3)
}  // namespace fused
}  // namespace reg
