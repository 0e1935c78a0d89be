// stage_rows_f64.cu -- advection row passes of the transport stages in double precision.
#include "stage_launch.cuh"

namespace reg {
namespace fused {
REG_ROWS_OF(double, EPI_ADV2)
REG_ROWS_OF(double, EPI_ADV3)
}  // namespace fused
}  // namespace reg
