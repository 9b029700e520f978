// kernels_f64_models.cu -- FP64 instantiations of the Gaussian-prior model,
// the LSQ-Wiener filter and the adjoint (a translation unit of their own, so
// that the FP64 kernels compile in parallel).
#include "launch.cuh"

namespace plc {
template void grad_newton_g<double, double, double>(plc_ctx*, const double*, const double*,
                                                    const int32_t*, double, double*, double*,
                                                    double*, double*, bool);
template void grad_newton_g<double, double, float>(plc_ctx*, const double*, const double*,
                                                   const int32_t*, double, double*, double*,
                                                   float*, float*, bool);
template void newton_update_g<double, double>(plc_ctx*, const double*, const double*,
                                              const double*, const double*, const double*,
                                              const double*, const int32_t*, const double*,
                                              double, double, bool, double*, double*, double*,
                                              double*, double*);
template void newton_update_g<double, float>(plc_ctx*, const double*, const double*,
                                             const double*, const float*, const float*,
                                             const float*, const int32_t*, const double*, double,
                                             double, bool, double*, double*, double*, float*,
                                             float*);
template void boundary_step<double, double>(plc_ctx*, const double*, const double*, const int32_t*);
template void boundary_step<double, float>(plc_ctx*, const double*, const float*, const int32_t*);
template void vjp_amplitude<double>(plc_ctx*, const double*, const double*);
template void diag_start_g<double>(plc_ctx*, double*, const int32_t*, const double*, double);
template void lsq_init<double>(plc_ctx*, const int32_t*, const double*, double, double*, double*,
                              bool);
}  // namespace plc
