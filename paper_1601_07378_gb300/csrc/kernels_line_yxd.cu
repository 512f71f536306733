// kernels_line_yxd.cu -- y/x pass of the line path, size class 48 to 96, n1 = 72, 80 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<1, 72>;
template struct LaunchYX<1, 80>;
}  // namespace line
}  // namespace vloc
