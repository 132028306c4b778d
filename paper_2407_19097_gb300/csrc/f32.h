// FP32 convolutions on NHWC tensors (f32.cu).
#pragma once
#include "internal.h"

namespace nrv {

// 3x3 "same" conv of concat(x1 [c1], x2 [c2]) with weights [tap][c][n]: bias (may be null), ReLU,
// then zero where mask (shaped like y; may be null) is not positive.  Also the data gradient of
// a 3x3 conv, given its rotated, transposed weights.
nrv_status f32_conv3(const float* x1, int c1, const float* x2, int c2, const float* w, const float* bias,
                     int relu, const float* mask, float* y, int cout, int n, int h, int wd, cudaStream_t s);
// 2x2 stride-2 transposed conv of x [n][h][wd][cin] to y [n][2h][2wd][cout], weights [ab][c][o].
nrv_status f32_upconv(const float* x, int cin, const float* w, const float* bias, float* y, int cout, int n,
                      int h, int wd, cudaStream_t s);
// Its data gradient from g at (2h, 2wd), ldg channels per pixel of which the first cout, weights
// [ab][o][c]; zero where mask (the layer's input) is not positive.
nrv_status f32_upconv_dgrad(const float* g, int ldg, int cout, const float* wt, const float* mask, float* gx,
                            int cin, int n, int h, int wd, cudaStream_t s);

// Weight and bias gradient partials of a 3x3 conv: part[split][o][tap * cin + c] and
// partb[split][o] over f32_wgrad_splits() splits of the pixels (g: [n][h][wd][cout]).
int f32_wgrad_splits(int cin, int cout, int n, int h, int wd);
nrv_status f32_wgrad(const float* g, int cout, const float* x1, int c1, const float* x2, int c2, int n, int h,
                     int wd, float* part, float* partb, cudaStream_t s);
// Of a transposed conv: part[split][c][ab * cout + o], partb[split][ab * cout + o]; g at (2h, 2wd)
// with ldg channels per pixel, of which the first cout.
int f32_wgrad_up_splits(int cin, int cout, int n, int h, int wd);
nrv_status f32_wgrad_up(const float* x, int cin, const float* g, int ldg, int cout, int n, int h, int wd,
                        float* part, float* partb, cudaStream_t s);

}  // namespace nrv
