// Instantiations of the float64 sweeps (fixed-point arithmetic) for some grid lengths.
#include "gp_internal.h"

namespace gp {
cudaError_t sweep_f64_8(const FixArgs& a, cudaStream_t s) { return FixLaunch<8>::launch(a, s); }
cudaError_t sweep_f64_12(const FixArgs& a, cudaStream_t s) { return FixLaunch<12>::launch(a, s); }
cudaError_t sweep_f64_16(const FixArgs& a, cudaStream_t s) { return FixLaunch<16>::launch(a, s); }
cudaError_t sweep_f64_24(const FixArgs& a, cudaStream_t s) { return FixLaunch<24>::launch(a, s); }
cudaError_t sweep_f64_32(const FixArgs& a, cudaStream_t s) { return FixLaunch<32>::launch(a, s); }
cudaError_t sweep_f64_48(const FixArgs& a, cudaStream_t s) { return FixLaunch<48>::launch(a, s); }
}  // namespace gp
