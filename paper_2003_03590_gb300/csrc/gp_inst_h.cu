// Instantiations of the float64 sweeps (fixed-point arithmetic) for some grid lengths.
#include "gp_internal.h"

namespace gp {
cudaError_t sweep_f64_96(const FixArgs& a, cudaStream_t s) { return FixLaunch<96>::launch(a, s); }
cudaError_t sweep_f64_192(const FixArgs& a, cudaStream_t s) { return FixLaunch<192>::launch(a, s); }
}  // namespace gp
