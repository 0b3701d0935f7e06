// The work-list kernels of gk_game.cuh.
#include "gk_game.cuh"

namespace gk {

WorklistKernel worklist_kernel(bool multi, bool spawn) {
    if (!multi) return spawn ? k_worklist<false, true> : k_worklist<false, false>;
    return spawn ? k_worklist<true, true> : k_worklist<true, false>;
}

int fill_worklist_columns() { return fill_columns(); }

}  // namespace gk
