// Instantiation unit of the short-pipeline kernels (see eval_kernel.cuh):
// Eager 1F1B, M < 2S-1.
#include "eval_kernel.cuh"

namespace pos {

pos_status eval_eager_short_1_14(const EvalParams &p, cudaStream_t s) {
    return launch_short_range<true, 1, 14, 4>(p, s);
}

}  // namespace pos
