// kernels_df_e.cu -- FP64-data chain kernels (double-float and native), lengths 144.
#include "kernels_df.cuh"

namespace vloc {
template struct LaunchF64<0, 144>;
template struct LaunchF64<1, 144>;
}  // namespace vloc
