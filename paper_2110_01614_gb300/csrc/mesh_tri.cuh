// Point-triangle geometry shared by the mesh-distance kernels.
#pragma once

#include <cuda_runtime.h>

namespace nsdf {

template <typename T>
struct V3 {
  T x, y, z;
};
template <typename T>
__device__ __forceinline__ V3<T> sub(V3<T> a, V3<T> b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
template <typename T>
__device__ __forceinline__ T dot(V3<T> a, V3<T> b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
template <typename T>
__device__ __forceinline__ V3<T> cross(V3<T> a, V3<T> b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// Products and sums of the triangle test, each rounding written out: every
// kernel that calls it gets the same bits for the same point and triangle.
__device__ __forceinline__ float dot_rn(V3<float> a, V3<float> b) {
  return __fmaf_rn(a.z, b.z, __fmaf_rn(a.y, b.y, __fmul_rn(a.x, b.x)));
}
__device__ __forceinline__ float det_rn(float a, float b, float c, float d) {   // a b - c d
  return __fmaf_rn(a, b, -__fmul_rn(c, d));
}
__device__ __forceinline__ V3<float> along_rn(V3<float> a, V3<float> e, float t) {   // a + t e
  return {__fmaf_rn(t, e.x, a.x), __fmaf_rn(t, e.y, a.y), __fmaf_rn(t, e.z, a.z)};
}

// Squared distance from p to triangle (a, b, c) by its Voronoi regions.
__device__ __forceinline__ float tri_dist2(V3<float> p, V3<float> a, V3<float> b, V3<float> c) {
  const V3<float> ab = sub(b, a), ac = sub(c, a), ap = sub(p, a);
  const float d1 = dot_rn(ab, ap), d2 = dot_rn(ac, ap);
  V3<float> q;
  if (d1 <= 0.f && d2 <= 0.f) {
    q = a;
  } else {
    const V3<float> bp = sub(p, b);
    const float d3 = dot_rn(ab, bp), d4 = dot_rn(ac, bp);
    if (d3 >= 0.f && d4 <= d3) {
      q = b;
    } else {
      const float vc = det_rn(d1, d4, d3, d2);
      if (vc <= 0.f && d1 >= 0.f && d3 <= 0.f) {
        q = along_rn(a, ab, d1 / (d1 - d3));
      } else {
        const V3<float> cp = sub(p, c);
        const float d5 = dot_rn(ab, cp), d6 = dot_rn(ac, cp);
        if (d6 >= 0.f && d5 <= d6) {
          q = c;
        } else {
          const float vb = det_rn(d5, d2, d1, d6);
          if (vb <= 0.f && d2 >= 0.f && d6 <= 0.f) {
            q = along_rn(a, ac, d2 / (d2 - d6));
          } else {
            const float va = det_rn(d3, d6, d5, d4);
            if (va <= 0.f && (d4 - d3) >= 0.f && (d5 - d6) >= 0.f) {
              q = along_rn(b, sub(c, b), (d4 - d3) / ((d4 - d3) + (d5 - d6)));
            } else {
              const float den = 1.f / __fadd_rn(__fadd_rn(va, vb), vc);
              q = along_rn(along_rn(a, ab, __fmul_rn(vb, den)), ac, __fmul_rn(vc, den));
            }
          }
        }
      }
    }
  }
  const V3<float> d = sub(p, q);
  return dot_rn(d, d);
}

template <typename T>
__device__ __forceinline__ T solid_angle(V3<T> p, V3<T> a, V3<T> b, V3<T> c) {
  const V3<T> A = sub(a, p), B = sub(b, p), C = sub(c, p);
  const T la = sqrt(dot(A, A)), lb = sqrt(dot(B, B)), lc = sqrt(dot(C, C));
  const T num = dot(A, cross(B, C));
  const T den = la * lb * lc + dot(A, B) * lc + dot(A, C) * lb + dot(B, C) * la;
  return T(2) * atan2(num, den);
}

// Points of the implicit grid: node (i, j, k) at lo + (i, j, k) * h, index
// i + N (j + N k).
struct GridPts {
  int n;
  float lo[3], h[3];
};

// Query point idx: an explicit float4, or a node of the grid when pts is null.
__device__ __forceinline__ V3<float> query_point(const float4 *__restrict__ pts, const GridPts &grid,
                                                 int64_t idx) {
  if (pts) {
    const float4 p = pts[idx];
    return {p.x, p.y, p.z};
  }
  const int64_t N = grid.n;
  return {grid.lo[0] + grid.h[0] * (float)(idx % N), grid.lo[1] + grid.h[1] * (float)((idx / N) % N),
          grid.lo[2] + grid.h[2] * (float)(idx / (N * N))};
}

// What the distance starts from: a point or triangle that no distance can be
// computed for (a NaN, an overflow) leaves it there, so the result is its root.
constexpr float kFarDist2 = 3.4e38f;

}  // namespace nsdf
