// bias_f64_ops.cu -- FP64 instantiations of the linear-bias operators (the
// Hessian-vector products and S^-1), apart from the density and gradient
// pipelines of bias_f64.cu so that the two compile in parallel.
#include "bias.cuh"
#include "bias.h"

namespace plc {
template void bias_prior<double, double>(plc_ctx*, const double*, double, double*);
template void bias_prior<double, float>(plc_ctx*, const float*, double, double*);
template void bias_cg_hv<double>(plc_ctx*, const double*, const double*, double*, const double*,
                                 const double*, const double*, double*, double*, double*, bool);
template void bias_hv<double>(plc_ctx*, const double*, const double*, const double*,
                              const double*, double*, double*, double*);
}  // namespace plc
