// Instantiations of the float64 sweeps (fixed-point arithmetic) for some grid lengths.
#include "gp_internal.h"

namespace gp {
cudaError_t sweep_f64_256(const FixArgs& a, cudaStream_t s) { return FixLaunch<256>::launch(a, s); }
}  // namespace gp
