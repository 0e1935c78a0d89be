// stage_f32.cu -- single precision instantiation of the transport stages.
#include "stage_launch.cuh"

namespace reg {
template <>
void adv_stage<float>(Spectral<float>& sp, const float* u, const fused::AdvEpi<float>& e, float* gx, float* gy) {
  fused::adv_stage_impl<float>(sp, u, e, gx, gy);
}
template <>
void adv2_stage<float>(Spectral<float>& sp, const float* uA, const fused::AdvEpi<float>& eA, const float* uB,
                     const fused::AdvEpi<float>& eB, float* const* Z) {
  fused::adv2_stage_impl<float>(sp, uA, eA, uB, eB, Z);
}
template <>
void div_stage<float>(Spectral<float>& sp, const float* lam, const float* a, const fused::DivEpi<float>& e, float* kx, float* ky) {
  fused::div_stage_impl<float>(sp, lam, a, e, kx, ky);
}

}  // namespace reg
