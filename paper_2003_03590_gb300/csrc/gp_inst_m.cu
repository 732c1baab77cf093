#include "gp_argle.cuh"

namespace gp {
template struct ArgleLaunch<512>;
}  // namespace gp
