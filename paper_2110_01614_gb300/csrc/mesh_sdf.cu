// Exact signed distance to a watertight triangle mesh: the ground truth a
// network is fitted to (Sec. 3.1) and the plain reference a cloth run can
// collide against.  Closed meshes of 192 faces and more go through the tree of
// mesh_tree.cu; this is the brute force for the others and the dispatch.
//
// Per point: unsigned distance = min over triangles of the distance to the
// triangle's closest point (barycentric Voronoi-region test: vertex, edge or
// face region); sign from the generalized winding number
// w = sum_t Omega_t / (4 pi), inside (negative, Sec. 3.2) when w > 1/2, with
// Omega_t from the Van Oosterom-Strackee formula.
//
// Triangles stream through shared memory in chunks; each thread owns one
// point: an explicit float4, or node (i, j, k) of a regular grid (i fastest)
// when the voxel baseline builds its grid.  w is accumulated in FP32; for points where that is not decisive
// (|w - 1/2| < 0.25, or distance < 1e-3 where one nearby triangle's solid
// angle is ill-conditioned) the warp recomputes w in FP64, all 32 lanes
// splitting the triangles of one such point at a time.

#include <mutex>

#include "mesh_tree.cuh"
#include "nsdf_internal.h"

namespace nsdf {
namespace {

constexpr int kThreads = 256;
constexpr int kChunk = 512;           // triangles per shared-memory chunk
constexpr float kInv4Pi = 0.0795774715459476679f;

struct TriChunk {
  float ax[kChunk], ay[kChunk], az[kChunk];
  float bx[kChunk], by[kChunk], bz[kChunk];
  float cx[kChunk], cy[kChunk], cz[kChunk];
};

// A face with a vertex index outside [0, nv) is replaced by a triangle
// collapsed onto a point 1e30 away: it is never the closest and its solid
// angle is zero, so it drops out without an out-of-bounds read.
__device__ void load_chunk(TriChunk &t, const float *__restrict__ V, int64_t nv,
                           const int32_t *__restrict__ F, int64_t f0, int64_t nf) {
  for (int i = threadIdx.x; i < kChunk; i += blockDim.x) {
    const int64_t f = f0 + i;
    if (f < nf) {
      const int64_t a = F[3 * f], b = F[3 * f + 1], c = F[3 * f + 2];
      if (a < 0 || b < 0 || c < 0 || a >= nv || b >= nv || c >= nv) {
        t.ax[i] = t.bx[i] = t.cx[i] = 1e30f;
        t.ay[i] = t.by[i] = t.cy[i] = 0.f;
        t.az[i] = t.bz[i] = t.cz[i] = 0.f;
        continue;
      }
      t.ax[i] = V[3 * a]; t.ay[i] = V[3 * a + 1]; t.az[i] = V[3 * a + 2];
      t.bx[i] = V[3 * b]; t.by[i] = V[3 * b + 1]; t.bz[i] = V[3 * b + 2];
      t.cx[i] = V[3 * c]; t.cy[i] = V[3 * c + 1]; t.cz[i] = V[3 * c + 2];
    }
  }
}

// kAfterTree: launched behind the tree's kernels, and without faces, so that nothing
// is written, where they have answered.  (As an early return the same test made the
// loop over the faces 5% slower.)
template <bool kAfterTree>
__global__ void __launch_bounds__(kThreads) mesh_sdf_kernel(const float *__restrict__ V, int64_t nv,
                                                            const int32_t *__restrict__ F,
                                                            int64_t nf, const float4 *__restrict__ pts,
                                                            int64_t n, float *__restrict__ out,
                                                            const GridPts grid,
                                                            const MeshTreeHeader *tree) {
  extern __shared__ float4 smem4[];
  TriChunk &tc = *reinterpret_cast<TriChunk *>(smem4);
  __shared__ double wacc[kThreads / 32][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  V3<float> p = {0.f, 0.f, 0.f};
  if (idx < n) p = query_point(pts, grid, idx);
  if (kAfterTree && mesh_tree_usable(tree)) nf = 0;
  float best = kFarDist2, wsum = 0.f;
  for (int64_t f0 = 0; f0 < nf; f0 += kChunk) {
    __syncthreads();
    load_chunk(tc, V, nv, F, f0, nf);
    __syncthreads();
    const int m = (int)((nf - f0) < kChunk ? (nf - f0) : kChunk);
    for (int i = 0; i < m; ++i) {
      const V3<float> a = {tc.ax[i], tc.ay[i], tc.az[i]};
      const V3<float> b = {tc.bx[i], tc.by[i], tc.bz[i]};
      const V3<float> c = {tc.cx[i], tc.cy[i], tc.cz[i]};
      best = fminf(best, tri_dist2(p, a, b, c));
      wsum += solid_angle<float>(p, a, b, c);
    }
  }
  const float dist = sqrtf(best);
  float w = wsum * kInv4Pi;
  const bool redo = (idx < n) && (fabsf(w - 0.5f) < 0.25f || dist < 1e-3f);
  // FP64 winding number for the undecided points of this CTA
  const int any = __syncthreads_or(redo ? 1 : 0);
  if (any) {
    const unsigned mask = __ballot_sync(0xffffffffu, redo);
    wacc[warp][lane] = 0.0;
    for (int64_t f0 = 0; f0 < nf; f0 += kChunk) {
      __syncthreads();
      load_chunk(tc, V, nv, F, f0, nf);
      __syncthreads();
      const int m = (int)((nf - f0) < kChunk ? (nf - f0) : kChunk);
      unsigned todo = mask;
      while (todo) {
        const int q = __ffs(todo) - 1;
        todo &= todo - 1;
        const V3<double> pq = {(double)__shfl_sync(0xffffffffu, p.x, q),
                               (double)__shfl_sync(0xffffffffu, p.y, q),
                               (double)__shfl_sync(0xffffffffu, p.z, q)};
        double part = 0.0;
        for (int i = lane; i < m; i += 32) {
          const V3<double> a = {tc.ax[i], tc.ay[i], tc.az[i]};
          const V3<double> b = {tc.bx[i], tc.by[i], tc.bz[i]};
          const V3<double> c = {tc.cx[i], tc.cy[i], tc.cz[i]};
          part += solid_angle<double>(pq, a, b, c);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) wacc[warp][q] += part;
      }
    }
    __syncwarp();
    if (redo) w = (float)(wacc[warp][lane] / (4.0 * 3.14159265358979323846));
  }
  if (idx < n && (!kAfterTree || nf > 0)) out[idx] = (w > 0.5f) ? -dist : dist;
}

// The tree's scratch comes from a stream-ordered pool of the library's own, one per
// device.  The device's default pool gives its memory back whenever the caller
// synchronises, and the next call would map it again: 180 us, more than a small call
// takes.  This one keeps up to kPoolKeep bytes between calls and is emptied when a
// context is destroyed (mesh_scratch_trim).
constexpr uint64_t kPoolKeep = uint64_t(64) << 20;
constexpr int kMaxDevices = 64;
std::mutex g_pool_mutex;
cudaMemPool_t g_pool[kMaxDevices] = {};

cudaMemPool_t scratch_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  if (!g_pool[dev]) {
    // another thread may be capturing a stream
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = kPoolKeep;
    if (cudaMemPoolCreate(&pool, &props) == cudaSuccess) {
      if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess)
        g_pool[dev] = pool;
      else
        cudaMemPoolDestroy(pool);
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
  }
  return g_pool[dev];
}

}  // namespace

void mesh_scratch_trim(int device) {
  if (device < 0 || device >= kMaxDevices) return;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  if (g_pool[device]) cudaMemPoolTrimTo(g_pool[device], 0);
}

cudaError_t launch_mesh_sdf(const float *verts, int64_t n_verts, const int32_t *faces,
                            int64_t n_faces, const float4 *pts, int64_t n, float *out, int grid_n,
                            const float *lo, const float *h, cudaStream_t s) {
  const size_t smem = sizeof(TriChunk);
  cudaError_t e = cudaFuncSetAttribute(mesh_sdf_kernel<false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mesh_sdf_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  GridPts g{};
  if (!pts) {
    g.n = grid_n;
    for (int c = 0; c < 3; ++c) {
      g.lo[c] = lo[c];
      g.h[c] = h[c];
    }
  }
  // The tree needs scratch memory, taken from the pool and given back behind the
  // kernels.  Without it (none left, or a stream that is being captured: the graph
  // stays free of allocations) the brute-force kernel answers alone.
  void *mem = nullptr;
  if (n_faces >= kTreeMinFaces && n_faces <= kTreeMaxFaces) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
      const cudaMemPool_t pool = scratch_pool();
      const size_t bytes = mesh_tree_bytes(n_faces, pts ? n : 0, pts ? 0 : n);
      if (!pool || cudaMallocFromPoolAsync(&mem, bytes, pool, s) != cudaSuccess) mem = nullptr;
    }
    if (!mem) cudaGetLastError();
  }
  if (mem) {
    e = launch_mesh_tree(verts, n_verts, faces, n_faces, pts, n, out, g, mem, s);
    if (e != cudaSuccess) {
      cudaFreeAsync(mem, s);
      return e;
    }
  }
  const int64_t blocks = (n + kThreads - 1) / kThreads;
  const auto brute = mem ? mesh_sdf_kernel<true> : mesh_sdf_kernel<false>;
  brute<<<(unsigned)blocks, kThreads, smem, s>>>(verts, n_verts, faces, n_faces, pts, n, out, g,
                                                 static_cast<const MeshTreeHeader *>(mem));
  e = cudaGetLastError();
  if (mem) {
    const cudaError_t e2 = cudaFreeAsync(mem, s);
    if (e == cudaSuccess) e = e2;
  }
  return e;
}

}  // namespace nsdf

extern "C" nsdf_status nsdf_mesh_sdf(const float *verts, int64_t n_verts, const int32_t *faces,
                                     int64_t n_faces, const float *pts, int64_t n, float *out_sdf,
                                     nsdf_stream stream) {
  if (n < 0 || n_verts < 0 || n_faces < 0) return NSDF_ERR_INVALID_ARG;
  if (n == 0) return NSDF_OK;
  if (!verts || !faces || !pts || !out_sdf || n_faces == 0 || n_verts < 3) return NSDF_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(pts) & 15u) != 0) return NSDF_ERR_MISALIGNED;
  if (!nsdf::device_memory(verts) || !nsdf::device_memory(faces) || !nsdf::device_memory(pts) ||
      !nsdf::device_memory(out_sdf))
    return NSDF_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  return nsdf::launch_mesh_sdf(verts, n_verts, faces, n_faces, reinterpret_cast<const float4 *>(pts),
                               n, out_sdf, 0, nullptr, nullptr, s) == cudaSuccess
             ? NSDF_OK
             : NSDF_ERR_CUDA;
}
