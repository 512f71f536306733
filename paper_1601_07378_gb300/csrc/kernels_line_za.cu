// kernels_line_za.cu -- z-passes of the line path, lengths VLOC_LINE_Z_A (kernels_line.h).
#include "kernels_line_z.cuh"

namespace vloc {
namespace line {
#define VLOC_CASE(N) template struct LaunchZ<N>;
VLOC_LINE_Z_A(VLOC_CASE)
#undef VLOC_CASE
}  // namespace line
}  // namespace vloc
