// sw_score_ck.cu -- the score pass's kernels with checkpoints
// (sw_score_kernel.cuh).
#include "sw_score_kernel.cuh"

namespace swgb {

const void *score_kernel_ck(int rows, int mode, bool fma) { return score_kernel_at<true>(rows, mode, fma); }

}  // namespace swgb
