// Many bodies in one launch (batching form): every network of a context
// answers its own range of points, all in one persistent grouped launch.
//
// The work list is built on the device from the counts, so a CUDA graph that
// captured nsdf_query_grouped replays correctly after the counts change:
// tile_start[k] = sum_{j<k} ceil(counts[j] / P), and tile t belongs to the
// network k with tile_start[k] <= t < tile_start[k+1].  The FP32 fused query
// kernel then walks the tiles persistently, fetching each tile's network
// weights from a device table of per-network pointers.  The tile shape and the
// CTAs per SM come from the context's tuned configuration (nsdf_autotune_grouped)
// or, without one, from the bodies' average size (query_fp32.cu).

#include "launch.cuh"
#include "nsdf_internal.h"

namespace nsdf {
namespace {

constexpr int kThreads = 256;

// T = [A | t; 0 0 0 1] (the last row is not read) gives the point map T^{-1} =
// [A^{-1} | -A^{-1} t] of Sec. 4.2, inverted in FP64 through the adjugate, and
// the normal rotation A.  A singular A is flagged and replaced by the identity.
__device__ void body_transform(const float *t, float *o, int *err) {
  const double a[9] = {t[0], t[1], t[2], t[4], t[5], t[6], t[8], t[9], t[10]};
  const double tx = t[3], ty = t[7], tz = t[11];
  // adjugate, row-major: adj[r][c] = cofactor of a[c][r]
  double adj[9] = {a[4] * a[8] - a[5] * a[7], a[2] * a[7] - a[1] * a[8], a[1] * a[5] - a[2] * a[4],
                   a[5] * a[6] - a[3] * a[8], a[0] * a[8] - a[2] * a[6], a[2] * a[3] - a[0] * a[5],
                   a[3] * a[7] - a[4] * a[6], a[1] * a[6] - a[0] * a[7], a[0] * a[4] - a[1] * a[3]};
  const double det = a[0] * adj[0] + a[1] * adj[3] + a[2] * adj[6];
  const bool ok = fabs(det) > 1e-30 && isfinite(det);
  if (!ok) atomicExch(err, kDevBadWork);
  for (int r = 0; r < 3; ++r) {
    double inv[3];
    for (int c = 0; c < 3; ++c) inv[c] = ok ? adj[r * 3 + c] / det : (r == c ? 1.0 : 0.0);
    o[r * 4 + 0] = (float)inv[0];
    o[r * 4 + 1] = (float)inv[1];
    o[r * 4 + 2] = (float)inv[2];
    o[r * 4 + 3] = ok ? (float)(-(inv[0] * tx + inv[1] * ty + inv[2] * tz)) : 0.f;
  }
  for (int i = 0; i < 9; ++i) o[12 + i] = ok ? (float)a[i] : (i % 4 == 0 ? 1.f : 0.f);
  for (int i = 21; i < kBodyFloats; ++i) o[i] = 0.f;
}

// One block prepares a grouped launch: the prefix sum of the networks' tile
// counts (at most a few thousand networks; a thread sums a run of them, the runs'
// sums are scanned) and, for posed scenes, every body's transform.  An entry
// outside [0, max_total) is dropped (zero tiles) and flagged.  Each network's tile
// count is rounded up to a multiple of `round_to` (the tensor-core kernels take
// tiles in pairs that must share a network).  One launch instead of two, and in
// parallel, and both it and the query overlap their predecessors' ends: a scene of
// 24 bodies and 59,000 points in FP16 32.6 -> 21.8 us, 3 posed bodies 34.1 -> 27.0.
__global__ void __launch_bounds__(kThreads) grouped_setup_kernel(
    const int64_t *offsets, const int64_t *counts, int n_nets, int P, int round_to, int64_t max_total,
    int32_t *tile_start, const float *T, float *body, int *err) {
  __shared__ int64_t sum[kThreads];
  wait_for_predecessor();
  release_successor();
  const int t = threadIdx.x;
  const int per = (n_nets + kThreads - 1) / kThreads, k0 = min(t * per, n_nets), k1 = min(k0 + per, n_nets);
  auto tiles_of = [&](int k) -> int64_t {
    const int64_t o = offsets[k], c = counts[k];
    if (c <= 0) return 0;
    if (o < 0 || o > max_total - c) {
      atomicExch(err, kDevBadWork);
      return 0;
    }
    return ((c + P - 1) / P + round_to - 1) / round_to * round_to;
  };
  int64_t own = 0;
  for (int k = k0; k < k1; ++k) own += tiles_of(k);
  sum[t] = own;
  for (int o = 1; o < kThreads; o <<= 1) {
    __syncthreads();
    const int64_t v = t >= o ? sum[t - o] : 0;
    __syncthreads();
    sum[t] += v;
  }
  int64_t acc = sum[t] - own;
  if (t == 0) tile_start[0] = 0;
  for (int k = k0; k < k1; ++k) {
    acc += tiles_of(k);
    tile_start[k + 1] = (int32_t)acc;
  }
  if (T)
    for (int k = t; k < n_nets; k += kThreads) body_transform(T + 16 * k, body + (size_t)kBodyFloats * k, err);
}

}  // namespace

cudaError_t launch_grouped_setup(const int64_t *offsets, const int64_t *counts, int n_nets, int P,
                                 int64_t max_total, int32_t *tile_start, int round_to, const float *T,
                                 float *body, int *err, cudaStream_t s) {
  return launch_overlapped(grouped_setup_kernel, dim3(1), kThreads, 0, s, offsets, counts, n_nets, P,
                           round_to, max_total, tile_start, T, body, err);
}

}  // namespace nsdf
