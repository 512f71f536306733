// kernels_line_yxa.cu -- y/x pass of the line path, size class up to 48, n1 = 24, 30, 32, 36, 40, 48 (kernels_line.h).
#include "kernels_line.cuh"

namespace vloc {
namespace line {
template struct LaunchYX<0, 24>;
template struct LaunchYX<0, 30>;
template struct LaunchYX<0, 32>;
template struct LaunchYX<0, 36>;
template struct LaunchYX<0, 40>;
template struct LaunchYX<0, 48>;
}  // namespace line
}  // namespace vloc
