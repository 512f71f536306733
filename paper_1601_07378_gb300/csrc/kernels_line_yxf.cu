// kernels_line_yxf.cu -- y/x pass of the line path, size class 80 to 144, n1 = 80, 90 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<2, 80>;
template struct LaunchYX<2, 90>;
}  // namespace line
}  // namespace vloc
