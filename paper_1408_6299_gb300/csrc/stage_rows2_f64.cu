// stage_rows2_f64.cu -- two-field and divergence row passes of the transport stages in double precision.
#include "stage_launch.cuh"

namespace reg {
namespace fused {
REG_ROWS_OF(double, EPI_ADV33)
REG_ROWS_OF(double, EPI_DIV)
}  // namespace fused
}  // namespace reg
