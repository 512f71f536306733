// kernels_line_yxg.cu -- y/x pass of the line path, size class 80 to 144, n1 = 96 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<2, 96>;
}  // namespace line
}  // namespace vloc
