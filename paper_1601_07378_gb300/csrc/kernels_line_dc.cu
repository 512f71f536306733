// kernels_line_dc.cu -- density of the line path, n1 = 80, 96, 100 (kernels_line.h).
#include "kernels_line_dens.cuh"

namespace vloc {
namespace line {
template struct LaunchDens<2, 80>;
template struct LaunchDens<2, 96>;
template struct LaunchDens<2, 100>;
}  // namespace line
}  // namespace vloc
