// The value function's split-digit path (masked_game_split.cu).
#pragma once

#include "tt_fsi.h"

namespace ttfsi_mgs {

// Whether the path takes a model of these sizes.
bool split_serves(int d, int h1, int h2, long long B, int out_f32);

// v[b, S] = mean over the n_bg rows of bg_dev of f(x_S, row elsewhere), all
// coalitions, float64 or (out_f32) float32; arguments already checked.
tt_fsi_status split_launch(const tt_fsi_mlp *model, const double *x_dev, const double *bg_dev, int n_bg, long long B,
                           void *v_dev, int out_f32, struct CUstream_st *stream);

}  // namespace ttfsi_mgs
