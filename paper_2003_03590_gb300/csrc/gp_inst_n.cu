#include "gp_argle.cuh"

namespace gp {
template struct ArgleLaunch<256>;
template struct ArgleLaunch<192>;
template struct ArgleLaunch<128>;
}  // namespace gp
