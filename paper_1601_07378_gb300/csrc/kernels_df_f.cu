// kernels_df_f.cu -- FP64-data chain kernels (double-float and native), lengths 96.
#include "kernels_df.cuh"

namespace vloc {
template struct LaunchF64<0, 96>;
template struct LaunchF64<1, 96>;
}  // namespace vloc
