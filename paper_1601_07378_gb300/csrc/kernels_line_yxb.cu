// kernels_line_yxb.cu -- y/x pass of the line path, size class 48 to 96, n1 = 48, 50, 54 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<1, 48>;
template struct LaunchYX<1, 50>;
template struct LaunchYX<1, 54>;
}  // namespace line
}  // namespace vloc
