// step_fast_ext.cu -- the double-float step with the options of the paper's
// experiments (exclusion, strategy (a), direct location) in the lean kernel,
// and the full node step alone (statistics, debug outputs, strategy (c)).
#include "step_lean_impl.cuh"

namespace sl {

void launch_lean_df_ext(const FastArgs &a, cudaStream_t s) { launch_lean_df_cfg<128, 8, true>(a, s); }

void launch_full_df(const FastArgs &a, bool stats, bool debug, cudaStream_t s)
{
    // (the plain form of the kernel counts or reports)
    if (a.exclude || a.order || a.grid_M > 0 || a.keep_t0 || !(stats || debug)) launch_fast_df_cfg<128, 8, true>(a, stats, debug, s);
    else launch_fast_df_cfg<128, 8>(a, stats, debug, s);
}

}  // namespace sl
