// kernels_line_yxi.cu -- y/x pass of the line path, size class 80 to 144, n1 = 108 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<2, 108>;
}  // namespace line
}  // namespace vloc
