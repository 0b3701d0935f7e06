// The multi-frame step kernels (resident rollouts) of gk_game.cuh.
#include "gk_game.cuh"

namespace gk {

StepKernel rollout_kernel(int lw, bool uniform, bool spawn) {
    if (spawn) return lw == 32 ? k_generals<true, true, 32, false> : k_generals<true, true, 16, false>;
    if (lw == 32) return uniform ? k_generals<true, false, 32, true> : k_generals<true, false, 32, false>;
    if (lw == 16) return uniform ? k_generals<true, false, 16, true> : k_generals<true, false, 16, false>;
    return uniform ? k_generals<true, false, 8, true> : k_generals<true, false, 8, false>;
}

int fill_rollout_columns() { return fill_columns(); }

}  // namespace gk
