#include "gp_argle.cuh"

namespace gp {
template struct ArgleLaunch<1024>;
}  // namespace gp
