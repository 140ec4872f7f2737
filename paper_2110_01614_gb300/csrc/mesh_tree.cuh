// Bounding-box tree over a triangle mesh (mesh_tree.cu), built on the device
// by every call that uses it.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "mesh_tri.cuh"

namespace nsdf {

// Written by the build, read by the queries.  All zero before the build.
struct MeshTreeHeader {
  unsigned neg_lo[3], hi[3];      // bounds of the faces kept, as ordered keys (neg_lo: of -lo)
  unsigned valid;                 // faces kept (every vertex index in range)
  unsigned nonfinite;             // a kept face has a NaN or infinite vertex
  unsigned long long boundary;    // hash of the mesh's boundary: 0 for a closed mesh
  unsigned done;                  // blocks of the box kernel that have finished
};

// Can the tree answer for this mesh?  Only a closed mesh of finite vertices
// has a winding number that ray crossings give.
__device__ __forceinline__ bool mesh_tree_usable(const MeshTreeHeader *h) {
  return h->boundary == 0ull && h->nonfinite == 0u && h->valid > 0u;
}

// Meshes below this take the brute-force kernel: far points, whose descents are
// long, cost more in a tree of so few faces than its eight launches and the descent
// save (128 faces, 8,000 and 30,000 points anywhere in the cube: 86 and 88 us by brute
// force, 103 and 109 through the tree; 192 faces: 125 and 127 against 123 and 131; 256:
// 165 and 166 against 133 and 140.  Points near the surface gain from 128 on).  Above
// the maximum 32-bit heap indices would run out.
constexpr int64_t kTreeMinFaces = 192;
constexpr int64_t kTreeMaxFaces = int64_t(1) << 28;

// n_points: explicit query points; n_nodes: nodes of a grid (the other is 0).
size_t mesh_tree_bytes(int64_t n_faces, int64_t n_points, int64_t n_nodes);
// Build the tree in `mem` (mesh_tree_bytes, 256-byte aligned) and write the
// signed distances of all points if it is usable; out is untouched otherwise.
cudaError_t launch_mesh_tree(const float *verts, int64_t n_verts, const int32_t *faces,
                             int64_t n_faces, const float4 *pts, int64_t n, float *out,
                             const GridPts &grid, void *mem, cudaStream_t s);

}  // namespace nsdf
