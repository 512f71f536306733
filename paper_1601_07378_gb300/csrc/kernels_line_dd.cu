// kernels_line_dd.cu -- density of the line path, n1 = 120, 128, 144 (kernels_line.h).
#include "kernels_line_dens.cuh"

namespace vloc {
namespace line {
template struct LaunchDens<2, 120>;
template struct LaunchDens<2, 128>;
template struct LaunchDens<2, 144>;
}  // namespace line
}  // namespace vloc
