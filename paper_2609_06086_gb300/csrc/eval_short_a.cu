// Instantiation unit of the short-pipeline kernels (see eval_kernel.cuh):
// 1F1B, M < S.
#include "eval_kernel.cuh"

namespace pos {

pos_status eval_short_1_9(const EvalParams &p, cudaStream_t s) {
    return launch_short_range<false, 1, 9, 4>(p, s);
}


pos_status eval_short_10_15(const EvalParams &p, cudaStream_t s) {
    return launch_short_range<false, 10, 15, 3>(p, s);
}

}  // namespace pos
