// The sliding-window factor in split FP32 (sympix_window.cuh).
#include "sympix_window.cuh"

namespace sympix {

void launch_window_df(sympix_plan_t pl, double *blocks, int32_t *info, cudaStream_t st) {
    launch_window_lists<DF>(pl, pl->win_one[SYMPIX_PREC_FP32X2], blocks, info, st);
}

}  // namespace sympix
