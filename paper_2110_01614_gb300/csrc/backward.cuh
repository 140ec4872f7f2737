// Launch parameters shared by the backward kernels (backward.cu for any shape
// that fits shared memory, backward_w64.cu for width 64).
#pragma once

#include "nsdf_internal.h"

namespace nsdf {

constexpr int kBwdMaxL = 16;

struct BwdParams {
  const float4 *pts;
  int64_t n;
  const float *a;        // [n]
  const float4 *v;       // [n] or null
  float *g_partial;      // [grid][n_params] or null
  float4 *g_pts;         // [n] or null
  const float *w0, *bias, *fwd_t, *bwd, *wout, *bout;
  int W, L, skip;
  float beta;
  int64_t n_params;
  int64_t woff[kBwdMaxL + 1], boff[kBwdMaxL + 1];
  int out[kBwdMaxL + 1];
};

// Width 64, two or three hidden layers.
bool backward_w64_supported(int width, int n_hidden);
cudaError_t launch_backward_w64(const BwdParams &p, int grid, cudaStream_t s);

}  // namespace nsdf
