// stage_f64.cu -- double precision instantiation of the transport stages.
#include "stage_launch.cuh"

namespace reg {
template <>
void adv_stage<double>(Spectral<double>& sp, const double* u, const fused::AdvEpi<double>& e, double* gx, double* gy) {
  fused::adv_stage_impl<double>(sp, u, e, gx, gy);
}
template <>
void adv2_stage<double>(Spectral<double>& sp, const double* uA, const fused::AdvEpi<double>& eA, const double* uB,
                     const fused::AdvEpi<double>& eB, double* const* Z) {
  fused::adv2_stage_impl<double>(sp, uA, eA, uB, eB, Z);
}
template <>
void div_stage<double>(Spectral<double>& sp, const double* lam, const double* a, const fused::DivEpi<double>& e, double* kx, double* ky) {
  fused::div_stage_impl<double>(sp, lam, a, e, kx, ky);
}

}  // namespace reg
