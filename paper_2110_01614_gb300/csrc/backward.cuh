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

// softplus_beta(z) and its slope to FP32 rounding: gradients of networks of any
// sharpness go through here (the hardware approximations that the query kernel takes
// err by up to 2^-21 / beta and lose log1p(e) altogether below e = 6e-8).
__device__ __forceinline__ void softplus_and_slope(float z, float beta, float &h, float &s) {
  const float e = expf(-beta * fabsf(z));
  h = fmaxf(z, 0.0f) + log1pf(e) / beta;
  const float inv = 1.0f / (1.0f + e);
  s = (z >= 0.0f) ? inv : e * inv;
}

// Width 64, two or three hidden layers.
bool backward_w64_supported(int width, int n_hidden);
cudaError_t launch_backward_w64(const BwdParams &p, int grid, cudaStream_t s);

}  // namespace nsdf
