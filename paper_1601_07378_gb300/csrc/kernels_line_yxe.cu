// kernels_line_yxe.cu -- y/x pass of the line path, size class 48 to 96, n1 = 90, 96 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<1, 90>;
template struct LaunchYX<1, 96>;
}  // namespace line
}  // namespace vloc
