// kernels_line_db.cu -- density of the line path, n1 = 72, 80, 96 (kernels_line.h).
#include "kernels_line_dens.cuh"

namespace vloc {
namespace line {
template struct LaunchDens<1, 72>;
template struct LaunchDens<1, 80>;
template struct LaunchDens<1, 96>;
}  // namespace line
}  // namespace vloc
