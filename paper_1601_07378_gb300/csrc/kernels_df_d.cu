// kernels_df_d.cu -- FP64-data chain kernels (double-float and native), lengths 120.
#include "kernels_df.cuh"

namespace vloc {
template struct LaunchF64<0, 120>;
template struct LaunchF64<1, 120>;
}  // namespace vloc
