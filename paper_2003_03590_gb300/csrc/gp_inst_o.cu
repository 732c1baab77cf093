#include "gp_argle.cuh"

namespace gp {
template struct ArgleLaunch<96>;
template struct ArgleLaunch<64>;
template struct ArgleLaunch<48>;
template struct ArgleLaunch<32>;
template struct ArgleLaunch<24>;
template struct ArgleLaunch<16>;
template struct ArgleLaunch<12>;
template struct ArgleLaunch<8>;
}  // namespace gp
