// kernels_line_yxk.cu -- y/x pass of the line path, size class 80 to 144, n1 = 128, 144 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<2, 128>;
template struct LaunchYX<2, 144>;
}  // namespace line
}  // namespace vloc
