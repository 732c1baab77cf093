// Instantiations of the float64 sweeps (fixed-point arithmetic) for some grid lengths.
#include "gp_internal.h"

namespace gp {
cudaError_t sweep_f64_64(const FixArgs& a, cudaStream_t s) { return FixLaunch<64>::launch(a, s); }
cudaError_t sweep_f64_128(const FixArgs& a, cudaStream_t s) { return FixLaunch<128>::launch(a, s); }
}  // namespace gp
