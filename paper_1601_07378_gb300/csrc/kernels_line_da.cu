// kernels_line_da.cu -- density of the line path, n1 = 32, 48, 48, 60, 64 (kernels_line.h).
#include "kernels_line_dens.cuh"

namespace vloc {
namespace line {
template struct LaunchDens<0, 32>;
template struct LaunchDens<0, 48>;
template struct LaunchDens<1, 48>;
template struct LaunchDens<1, 60>;
template struct LaunchDens<1, 64>;
}  // namespace line
}  // namespace vloc
