// One explicit Verlet step of a rectangular quad cloth (Sec. 4.1).
//
// Each thread owns one vertex and gathers the Hooke forces of its (up to)
// eight springs from the implicit grid topology: four structural neighbours
// (rest lengths hx along a row, hz between rows) and four shear neighbours
// (rest length sqrt(hx^2 + hz^2)).  Unit mass:
//   x_new = 2 x - x_prev + dt^2 (sum_j k (|d_j| - r_j) d_j/|d_j| + (0, -g, 0)).
// Gathering per vertex needs no atomics; every spring is evaluated from both
// ends, with equal and opposite results.  x_new overwrites x_prev in place
// (each thread reads and writes only its own x_prev entry).
//
// Bound: instruction issue and memory alike (48 B per vertex, 50 MB at 1024 x
// 1024: 7.4 us at 6.8 TB/s).  With an IEEE square root and division per spring
// (about 60 instructions of 590 per vertex) the issue slots were 77% busy; the
// approximate reciprocal root with a residual step for the length and one for the
// quotient needs 16 and rounds alike (the same bits on 1024 x 1024 random cloths).
// 1024 x 1024, x and x_prev from DRAM: 20.5 -> 14.9 us launched overlapped (14.1 with
// 1 - rest / |d| from the reciprocal alone, which leaves a force on springs at rest);
// tiles of 32 x 8 vertices read 1.3 rows per row written.  Evaluating each spring once,
// in strips that pass the scalars on by shuffles, measured 15.5 us against 12.4 with
// everything in L2: the shuffles and the lower occupancy cost more than the springs.

#include "launch.cuh"
#include "nsdf_internal.h"

namespace nsdf {
namespace {

constexpr int kTileX = 32, kTileY = 8;

// k (|d| - rest) / |d|, 0 for a spring of no length.  The length by a Newton step on
// its residual, so that a spring at rest gives exactly 0, and so the quotient.
__device__ __forceinline__ float spring(float dx, float dy, float dz, float rest, float k) {
  const float d2 = dx * dx + dy * dy + dz * dz;
  const float r = rsqrtf(d2), l = d2 * r;
  const float len = fmaf(0.5f * r, fmaf(-l, l, d2), l);
  const float a = k * (len - rest), q = a * r;
  return d2 > 0.f ? fmaf(fmaf(-q, len, a), r, q) : 0.f;
}

// (Plain pointers: an invariant load might move ahead of the wait.)
__global__ void __launch_bounds__(kTileX *kTileY) cloth_step_kernel(const float4 *x, float4 *xprev,
                                                                    int nx, int ny, float hx, float hz,
                                                                    float k, float g, float dt) {
  const int j = blockIdx.x * kTileX + threadIdx.x % kTileX;   // column (along x)
  const int i = blockIdx.y * kTileY + threadIdx.x / kTileX;   // row (along z)
  wait_for_predecessor();
  release_successor();
  if (j >= nx || i >= ny) return;
  const int64_t v = (int64_t)i * nx + j;
  const float4 p = x[v], pp = xprev[v];
  const float hd = sqrtf(hx * hx + hz * hz);
  float ax = 0.f, ay = -g, az = 0.f;
  const int di[8] = {0, 0, -1, 1, -1, -1, 1, 1};
  const int dj[8] = {-1, 1, 0, 0, -1, 1, -1, 1};
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int ii = i + di[s], jj = j + dj[s];
    if (ii < 0 || ii >= ny || jj < 0 || jj >= nx) continue;
    const float rest = s < 2 ? hx : (s < 4 ? hz : hd);
    const float4 q = x[(int64_t)ii * nx + jj];
    const float dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
    const float f = spring(dx, dy, dz, rest, k);
    ax = fmaf(f, dx, ax); ay = fmaf(f, dy, ay); az = fmaf(f, dz, az);
  }
  const float dt2 = dt * dt;
  float4 o;
  o.x = 2.f * p.x - pp.x + dt2 * ax;
  o.y = 2.f * p.y - pp.y + dt2 * ay;
  o.z = 2.f * p.z - pp.z + dt2 * az;
  o.w = p.w;
  xprev[v] = o;
}

}  // namespace
}  // namespace nsdf

extern "C" nsdf_status nsdf_cloth_step(const float *x, float *x_prev_inout, int nx, int ny, float hx,
                                       float hz, float k_over_m, float g, float dt,
                                       nsdf_stream stream) {
  if (nx < 0 || ny < 0 || !(hx > 0.f) || !(hz > 0.f) || !(dt > 0.f)) return NSDF_ERR_INVALID_ARG;
  if (nx == 0 || ny == 0) return NSDF_OK;
  if (!x || !x_prev_inout || x == x_prev_inout || ny > 65535 || nx > (1 << 30))
    return NSDF_ERR_INVALID_ARG;   // grid.y limit; the column index stays an int
  if ((reinterpret_cast<uintptr_t>(x) & 15u) || (reinterpret_cast<uintptr_t>(x_prev_inout) & 15u))
    return NSDF_ERR_MISALIGNED;
  if (!nsdf::device_memory(x) || !nsdf::device_memory(x_prev_inout)) return NSDF_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const dim3 grid((unsigned)((nx + nsdf::kTileX - 1) / nsdf::kTileX),
                  (unsigned)((ny + nsdf::kTileY - 1) / nsdf::kTileY));
  return nsdf::launch_overlapped(nsdf::cloth_step_kernel, grid, nsdf::kTileX * nsdf::kTileY, 0, s,
                                 reinterpret_cast<const float4 *>(x),
                                 reinterpret_cast<float4 *>(x_prev_inout), nx, ny, hx, hz, k_over_m,
                                 g, dt) == cudaSuccess
             ? NSDF_OK
             : NSDF_ERR_CUDA;
}
