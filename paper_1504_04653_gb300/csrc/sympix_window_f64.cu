// The sliding-window factor in FP64 (sympix_window.cuh), and the launcher of
// both arithmetics.
#include "sympix_window.cuh"

namespace sympix {

void launch_window_f64(sympix_plan_t pl, double *blocks, int32_t *info, cudaStream_t st) {
    launch_window_lists<double>(pl, pl->win_one[SYMPIX_PREC_FP64], blocks, info, st);
}

void launch_window(sympix_plan_t pl, int precision, double *blocks, int32_t *info, cudaStream_t st) {
    if (pl->d_win[0].n > 0) {
        if (precision == SYMPIX_PREC_FP64)
            launch_window_f64(pl, blocks, info, st);
        else
            launch_window_df(pl, blocks, info, st);
        trace_mark(pl, st, precision == SYMPIX_PREC_FP64 ? "k_f64_window" : "k_df_window");
    }
    if (precision == SYMPIX_PREC_FP64)
        launch_band<ArF64>(pl, false, blocks, info, st, 0, true);  // 12 < w <= 16
    else
        launch_band<ArF2>(pl, false, blocks, info, st, 0, true);
    trace_mark(pl, st, "k_factor_band");
}

}  // namespace sympix
