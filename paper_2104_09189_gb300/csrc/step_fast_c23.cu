// step_fast_c23.cu -- launch configurations 2 and 3 of the double-float step kernel
// (a translation unit of their own, so that the configurations compile in
// parallel).
#include "step_lean_impl.cuh"

namespace sl {

void launch_lean_df_c2(const FastArgs &a, cudaStream_t s) { launch_lean_df_cfg<128, 8>(a, s); }

void launch_lean_df_c3(const FastArgs &a, cudaStream_t s) { launch_lean_df_cfg<128, 9>(a, s); }

}  // namespace sl
