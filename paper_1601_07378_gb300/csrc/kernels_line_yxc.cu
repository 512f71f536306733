// kernels_line_yxc.cu -- y/x pass of the line path, size class 48 to 96, n1 = 60, 64 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<1, 60>;
template struct LaunchYX<1, 64>;
}  // namespace line
}  // namespace vloc
