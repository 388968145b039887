// step_fast_c01.cu -- launch configurations 0 and 1 of the double-float step kernel
// (a translation unit of their own, so that the configurations compile in
// parallel).
#include "step_lean_impl.cuh"

namespace sl {

void launch_lean_df_c0(const FastArgs &a, cudaStream_t s) { launch_lean_df_cfg<256, 4>(a, s); }

void launch_lean_df_c1(const FastArgs &a, cudaStream_t s) { launch_lean_df_cfg<128, 16>(a, s); }

}  // namespace sl
