// stage_rows2_f32.cu -- two-field and divergence row passes of the transport stages in single precision.
#include "stage_launch.cuh"

namespace reg {
namespace fused {
REG_ROWS_OF(float, EPI_ADV33)
REG_ROWS_OF(float, EPI_DIV)
}  // namespace fused
}  // namespace reg
