// step_fast_c45.cu -- launch configurations 4 and 5 of the double-float step kernel
// (a translation unit of their own, so that the configurations compile in
// parallel).
#include "step_lean_impl.cuh"

namespace sl {

void launch_lean_df_c4(const FastArgs &a, cudaStream_t s) { launch_lean_df_cfg<256, 5>(a, s); }

void launch_lean_df_c5(const FastArgs &a, cudaStream_t s) { launch_lean_df_cfg<128, 12>(a, s); }

}  // namespace sl
