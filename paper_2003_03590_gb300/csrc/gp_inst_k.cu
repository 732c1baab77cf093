// Instantiations of the float64 sweeps (fixed-point arithmetic) for some grid lengths.
#include "gp_internal.h"

namespace gp {
cudaError_t sweep_f64_1024(const FixArgs& a, cudaStream_t s) { return FixLaunch<1024>::launch(a, s); }
}  // namespace gp
