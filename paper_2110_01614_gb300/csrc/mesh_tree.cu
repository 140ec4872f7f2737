// Exact signed distance to a closed triangle mesh through a bounding-box tree.
//
// The brute-force kernel (mesh_sdf.cu) evaluates every point against every
// triangle.  Both halves of its answer need only a few of them:
//   * distance: the closest triangle, found by descending a tree of axis-
//     aligned boxes nearest first and skipping a box that lies further than
//     the best distance so far.  The triangle test is the brute-force one, and
//     a box is skipped only when it is further by more than the rounding of
//     that test, so the minimum is taken over the same triangle.
//   * sign: w > 1/2 for the generalized winding number w.  The mesh is closed
//     when its oriented edges cancel in pairs; then w is a whole number and
//     equals the signed count of the triangles that a ray from the point
//     crosses, along any axis (the one towards the nearest side of the mesh's
//     box, which meets the fewest boxes).  A triangle is crossed when the
//     projected point has a nonzero 2-D winding number about the projected
//     triangle, with one half-open rule and one evaluation order for each
//     edge, so that the triangles on either side of an edge always agree and
//     no crossing is lost or counted twice.  Side tests that FP32 does not
//     settle beyond its rounding are FP64.
// In front of either test of a triangle stands one of its bounding sphere.
// Closedness is tested on the device by a hash of the boundary: every oriented
// edge (a, b), named by the positions of its ends, adds h(a, b) - h(b, a)
// modulo 2^64.  A closed mesh gives exactly 0; any other gives 0 with
// probability about 2^-64.  A mesh that is not closed, or has a NaN or
// infinite vertex, is left to the brute-force kernel (the caller launches it
// next; it returns at once when the tree has answered).
//
// Build, per call, in scratch memory: bounds and hash (one pass over the
// faces), counting sort by the Morton cell of the centroid, leaves of four
// triangles, boxes of an implicit complete binary tree over the leaves, and
// the points' Morton order.  About 50 us for 20,480 triangles and 250,000
// points, so it is rebuilt by every call and nothing is kept between calls.
//
// Bound: instruction issue of the searches (60% and 41% of the slots in the two
// kernels) and their divergence (10 and 21 of 32 lanes active).  Measured on
// 250,000 fitting points (80% within 0.01 of the surface) and 20,480 triangles:
// brute force 107 ms; a thread per point in the caller's order with FP64 side
// tests 3.5 ms; hard points by their own warp, points in Morton order, FP32 filters
// 2.37 ms; spheres before the triangle tests and rays to the nearest side 2.1 ms;
// hard points from a list, four warps each 0.96 ms (Morton order had put them
// all into a few warps); one warp each where the list is long 0.87 ms.

#include "mesh_tree.cuh"

#include "nsdf_internal.h"

namespace nsdf {
namespace {

constexpr int kLeaf = 4;                 // triangles per leaf
constexpr int kBlock = 256;              // threads of the build kernels = leaves per box block
constexpr int kStack = 32;               // deeper than any tree of kTreeMaxFaces
constexpr int kPointBits = 5;            // Morton bits per axis of the points' order
constexpr int64_t kPointChunk = int64_t(1) << 20;
constexpr int64_t kHardMax = int64_t(1) << 18;
constexpr int kHardWarps = 4;            // warps that search one hard point
constexpr int kHardPerSm = 10;           // blocks that search hard points: as many as are resident
// Leaves a thread visits before its point is a hard one: 32 where points fill
// the GPU (6 / 12 / 20 / 32 measured 1.54 / 1.22 / 0.99 / 0.89 ms on 250,000
// fitting points, 48 and 96 more on far points), 4 where one thread's descent is all
// that a launch waits for (4 / 12 / 32: 200 points x 20,480 triangles 215 / 275 / 389
// us, 4,000 points 240 / 274 / 364 us).  The line is drawn at so many points per
// block of the hard kernel (48,640 here; 32 -> 4, far points: 8,000 points x 192
// triangles 173 -> 123 us, x 20,480 451 -> 274; 30,000 points x 320 193 -> 123; near
// ones 30,000 x 20,480 300 -> 259, x 320 100 -> 105; at 60,000 near points lose 8-19%).
constexpr int kLeafBudget = 32, kLeafBudgetFew = 4, kFewPerBlock = 32;

// Scratch layout for a mesh of F faces.
struct TreeMem {
  int64_t leaves;                        // power of two >= 2
  int bits;                              // Morton bits per axis
  int64_t chunk;                         // points ordered (and queried) at a time
  size_t header, hard_count, hist, phist, key, pkey, order, hard, tri, sphere, node, block_box, total;
  unsigned hard_cap;                     // points the hard list holds
};

__host__ inline TreeMem tree_mem(int64_t F, int64_t points, int64_t nodes) {
  TreeMem m{};
  m.chunk = points < kPointChunk ? points : kPointChunk;
  m.leaves = 2;
  while (m.leaves * kLeaf < F) m.leaves <<= 1;
  m.bits = F <= (int64_t(1) << 16) ? 5 : (F <= (int64_t(1) << 20) ? 6 : 7);
  size_t at = 0;
  auto take = [&at](size_t bytes) {
    const size_t o = at;
    at += (bytes + 255) & ~size_t(255);
    return o;
  };
  m.header = take(sizeof(MeshTreeHeader));
  m.hard_count = take(sizeof(unsigned));
  m.phist = take(m.chunk > 0 ? sizeof(unsigned) << (3 * kPointBits) : 0);
  m.hist = take(sizeof(unsigned) << (3 * m.bits));     // one memset clears these four
  m.key = take(sizeof(uint2) * (size_t)F);
  m.pkey = take(sizeof(uint2) * (size_t)m.chunk);
  m.order = take(sizeof(unsigned) * (size_t)m.chunk);
  const int64_t most = points > 0 ? m.chunk : nodes;
  m.hard_cap = (unsigned)(most < kHardMax ? most : kHardMax);
  m.hard = take(sizeof(int64_t) * (size_t)m.hard_cap);
  m.tri = take(sizeof(float4) * 3 * kLeaf * (size_t)m.leaves);
  m.sphere = take(sizeof(float4) * kLeaf * (size_t)m.leaves);
  m.node = take(sizeof(float4) * 3 * (size_t)m.leaves);
  const size_t blocks = (size_t)((m.leaves + kBlock - 1) / kBlock);
  m.block_box = take(sizeof(float) * 6 * 2 * blocks);
  m.total = at;
  return m;
}

// Order-preserving map of floats to unsigned.
__device__ __forceinline__ unsigned ordered(float f) {
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// splitmix64's finaliser (Steele, Lea & Flood, OOPSLA 2014).
__device__ __forceinline__ unsigned long long mix(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ unsigned long long vertex_key(V3<float> v) {
  // + 0.0f: the two zeros are one position
  const unsigned long long x = __float_as_uint(v.x + 0.0f), y = __float_as_uint(v.y + 0.0f),
                           z = __float_as_uint(v.z + 0.0f);
  return mix(mix((x << 32 | y) + 0x9e3779b97f4a7c15ull) ^ (z + 0xd1b54a32d192ed03ull));
}
__device__ __forceinline__ unsigned long long edge_term(unsigned long long a, unsigned long long b) {
  return mix(a * 0x9e3779b97f4a7c15ull + mix(b)) - mix(b * 0x9e3779b97f4a7c15ull + mix(a));
}

// The vertices of face f; false when an index lies outside [0, nv).
__device__ __forceinline__ bool load_face(const float *__restrict__ V, int64_t nv,
                                          const int32_t *__restrict__ F, int64_t f, V3<float> &a,
                                          V3<float> &b, V3<float> &c) {
  const int64_t i = F[3 * f], j = F[3 * f + 1], k = F[3 * f + 2];
  if (i < 0 || j < 0 || k < 0 || i >= nv || j >= nv || k >= nv) return false;
  a = {V[3 * i], V[3 * i + 1], V[3 * i + 2]};
  b = {V[3 * j], V[3 * j + 1], V[3 * j + 2]};
  c = {V[3 * k], V[3 * k + 1], V[3 * k + 2]};
  return true;
}

// Bounds, count, finiteness and boundary hash of the faces that are kept.
__global__ void __launch_bounds__(kBlock) tree_bounds_kernel(const float *__restrict__ V, int64_t nv,
                                                             const int32_t *__restrict__ F,
                                                             int64_t nf, MeshTreeHeader *hdr) {
  unsigned key[6] = {0u, 0u, 0u, 0u, 0u, 0u};
  unsigned valid = 0u, bad = 0u;
  unsigned long long hash = 0ull;
  for (int64_t f = (int64_t)blockIdx.x * kBlock + threadIdx.x; f < nf;
       f += (int64_t)gridDim.x * kBlock) {
    V3<float> a, b, c;
    if (!load_face(V, nv, F, f, a, b, c)) continue;
    ++valid;
    const float lo[3] = {fminf(fminf(a.x, b.x), c.x), fminf(fminf(a.y, b.y), c.y),
                         fminf(fminf(a.z, b.z), c.z)};
    const float hi[3] = {fmaxf(fmaxf(a.x, b.x), c.x), fmaxf(fmaxf(a.y, b.y), c.y),
                         fmaxf(fmaxf(a.z, b.z), c.z)};
    const float sum = (fabsf(a.x) + fabsf(a.y) + fabsf(a.z)) + (fabsf(b.x) + fabsf(b.y) + fabsf(b.z)) +
                      (fabsf(c.x) + fabsf(c.y) + fabsf(c.z));
    if (!(sum < 3.0e38f)) bad = 1u;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      key[k] = max(key[k], ordered(-lo[k]));
      key[3 + k] = max(key[3 + k], ordered(hi[k]));
    }
    const unsigned long long ka = vertex_key(a), kb = vertex_key(b), kc = vertex_key(c);
    hash += edge_term(ka, kb) + edge_term(kb, kc) + edge_term(kc, ka);
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) key[k] = __reduce_max_sync(0xffffffffu, key[k]);
  valid = __reduce_add_sync(0xffffffffu, valid);
  bad = __reduce_or_sync(0xffffffffu, bad);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hash += __shfl_xor_sync(0xffffffffu, hash, o);
  if ((threadIdx.x & 31) == 0 && valid) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      atomicMax(&hdr->neg_lo[k], key[k]);
      atomicMax(&hdr->hi[k], key[3 + k]);
    }
    atomicAdd(&hdr->valid, valid);
    if (bad) atomicOr(&hdr->nonfinite, 1u);
    atomicAdd(&hdr->boundary, hash);
  }
}

__device__ __forceinline__ unsigned spread3(unsigned v) {   // bits 0..6 to every third place
  unsigned r = 0u;
#pragma unroll
  for (int i = 0; i < 7; ++i) r |= ((v >> i) & 1u) << (3 * i);
  return r;
}

// Morton cell of position x on a grid of 2^bits cells along the longest side
// of the mesh's box (widened by `margin` of that side all round).
__device__ __forceinline__ unsigned cell_of(V3<float> x, const MeshTreeHeader *__restrict__ hdr,
                                            int bits, float margin) {
  float ext = 0.f, lo[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    lo[k] = -unordered(hdr->neg_lo[k]);
    ext = fmaxf(ext, unordered(hdr->hi[k]) - lo[k]);
  }
  const float cells = (float)(1 << bits);
  const float scale = cells / fmaxf(ext * (1.f + 2.f * margin), 1e-37f);
  const float c[3] = {x.x, x.y, x.z};
  unsigned m = 0u;
#pragma unroll
  for (int k = 0; k < 3; ++k)      // (a NaN goes to cell 0)
    m |= spread3((unsigned)fminf(fmaxf((c[k] - lo[k] + ext * margin) * scale, 0.f), cells - 1.f)) << k;
  return m;
}

// Counting sort, first pass: cell of each face (its centroid) and of each
// point, and its rank in the cell.  The first `fb` blocks take the faces.
__global__ void __launch_bounds__(kBlock) tree_cell_kernel(const float *__restrict__ V, int64_t nv,
                                                           const int32_t *__restrict__ F, int64_t nf,
                                                           int bits, unsigned fb,
                                                           const float4 *__restrict__ pts, int64_t n,
                                                           const MeshTreeHeader *__restrict__ hdr,
                                                           unsigned *hist, uint2 *__restrict__ key,
                                                           unsigned *phist, uint2 *__restrict__ pkey) {
  if (!mesh_tree_usable(hdr)) return;      // (here and below: an open mesh is not built)
  if (blockIdx.x >= fb) {
    const int64_t i = (int64_t)(blockIdx.x - fb) * kBlock + threadIdx.x;
    if (i >= n) return;
    const float4 p = pts[i];
    const unsigned m = cell_of({p.x, p.y, p.z}, hdr, kPointBits, 0.25f);
    pkey[i] = make_uint2(m, atomicAdd(&phist[m], 1u));
    return;
  }
  const int64_t f = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  if (f >= nf) return;
  V3<float> a, b, c;
  if (!load_face(V, nv, F, f, a, b, c)) {
    key[f] = make_uint2(0xffffffffu, 0u);
    return;
  }
  const unsigned m = cell_of({(a.x + b.x + c.x) * (1.f / 3.f), (a.y + b.y + c.y) * (1.f / 3.f),
                              (a.z + b.z + c.z) * (1.f / 3.f)},
                             hdr, bits, 0.f);
  key[f] = make_uint2(m, atomicAdd(&hist[m], 1u));
}

// Exclusive prefix sums of the cell counts, in place: block 0 the faces',
// block 1 the points'.  32 cells per thread and round (2^15 cells in one).
__global__ void __launch_bounds__(1024) tree_scan_kernel(const MeshTreeHeader *__restrict__ hdr,
                                                         unsigned *hist, int cells, unsigned *phist,
                                                         int pcells) {
  __shared__ unsigned warp_sum[32];
  if (!mesh_tree_usable(hdr)) return;
  if (blockIdx.x == 1) {
    hist = phist;
    cells = pcells;
  }
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  unsigned carry = 0u;
  for (int base = 0; base < cells; base += 32768) {
    uint4 *p = reinterpret_cast<uint4 *>(hist + base + 32 * t);
    uint4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = p[i];
    unsigned own = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) own += v[i].x + v[i].y + v[i].z + v[i].w;
    unsigned s = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned x = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += x;
    }
    if (lane == 31) warp_sum[w] = s;
    __syncthreads();
    // every warp sums the warps before it (and all of them, for the carry)
    const unsigned x = warp_sum[lane];
    const unsigned before = __reduce_add_sync(0xffffffffu, lane < w ? x : 0u);
    const unsigned all = __reduce_add_sync(0xffffffffu, x);
    unsigned e = carry + before + s - own;
    carry += all;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      uint4 r;
      r.x = e; e += v[i].x; r.y = e; e += v[i].y; r.z = e; e += v[i].z; r.w = e; e += v[i].w;
      p[i] = r;
    }
    __syncthreads();
  }
}

// Counting sort, second pass: faces into the leaves in cell order (three float4
// per triangle: a, b, c in turn), and the order in which the points are queried.
__global__ void __launch_bounds__(kBlock) tree_scatter_kernel(
    const float *__restrict__ V, int64_t nv, const int32_t *__restrict__ F, int64_t nf, unsigned fb,
    int64_t n, const MeshTreeHeader *__restrict__ hdr, const unsigned *__restrict__ start,
    const uint2 *__restrict__ key,
    const unsigned *__restrict__ pstart, const uint2 *__restrict__ pkey, float4 *__restrict__ tri,
    unsigned *__restrict__ order) {
  if (!mesh_tree_usable(hdr)) return;
  if (blockIdx.x >= fb) {
    const int64_t i = (int64_t)(blockIdx.x - fb) * kBlock + threadIdx.x;
    if (i >= n) return;
    const uint2 kr = pkey[i];
    order[pstart[kr.x] + kr.y] = (unsigned)i;
    return;
  }
  const int64_t f = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  if (f >= nf) return;
  const uint2 kr = key[f];
  if (kr.x == 0xffffffffu) return;
  V3<float> a, b, c;
  load_face(V, nv, F, f, a, b, c);
  float4 *o = tri + 3 * (size_t)(start[kr.x] + kr.y);
  o[0] = make_float4(a.x, a.y, a.z, b.x);
  o[1] = make_float4(b.y, b.z, c.x, c.y);
  o[2] = make_float4(c.z, 0.f, 0.f, 0.f);
}

struct Tri {
  V3<float> a, b, c;
};
__device__ __forceinline__ Tri load_tri(const float4 *__restrict__ t) {
  const float4 u = t[0], v = t[1], w = t[2];
  return {{u.x, u.y, u.z}, {u.w, v.x, v.y}, {v.z, v.w, w.x}};
}

struct Box {
  float lo[3], hi[3];
};
__device__ __forceinline__ Box join(const Box &a, const Box &b) {
  Box r;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.lo[k] = fminf(a.lo[k], b.lo[k]);
    r.hi[k] = fmaxf(a.hi[k], b.hi[k]);
  }
  return r;
}
// Node i of the heap order holds the boxes of its children 2i and 2i + 1.
__device__ __forceinline__ void store_node(float4 *node, int64_t i, const Box &l, const Box &r) {
  float4 *n = node + 3 * i;
  n[0] = make_float4(l.lo[0], l.lo[1], l.lo[2], l.hi[0]);
  n[1] = make_float4(l.hi[1], l.hi[2], r.lo[0], r.lo[1]);
  n[2] = make_float4(r.lo[2], r.hi[0], r.hi[1], r.hi[2]);
}

// Boxes bottom-up: each block reduces 256 leaves (a subtree) in shared memory,
// and the last block to finish builds the levels above the blocks' roots.
__global__ void __launch_bounds__(kBlock) tree_box_kernel(const float4 *__restrict__ tri,
                                                          float4 *__restrict__ sphere,
                                                          float4 *__restrict__ node, int leaves,
                                                          float *block_box, MeshTreeHeader *hdr) {
  __shared__ Box sb[kBlock];
  __shared__ bool last;
  if (!mesh_tree_usable(hdr)) return;
  const int t = threadIdx.x;
  const int per = leaves < kBlock ? leaves : kBlock;       // leaves of this block
  const int64_t leaf = (int64_t)blockIdx.x * per + t;
  Box b;
#pragma unroll
  for (int k = 0; k < 3; ++k) { b.lo[k] = INFINITY; b.hi[k] = -INFINITY; }
  const unsigned valid = hdr->valid;
  if (t < per) {
    for (int i = 0; i < kLeaf; ++i) {
      const int64_t f = leaf * kLeaf + i;
      if (f >= valid) {                  // padding: a NaN is never near and never crossed
        sphere[f] = make_float4(NAN, NAN, NAN, NAN);
        continue;
      }
      const Tri q = load_tri(tri + 3 * f);
      const float x[3][3] = {{q.a.x, q.b.x, q.c.x}, {q.a.y, q.b.y, q.c.y}, {q.a.z, q.b.z, q.c.z}};
      // centre of the triangle's box, and the furthest vertex from it (a little
      // further, for the rounding of the distances)
      float c[3], r2 = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float l = fminf(fminf(x[k][0], x[k][1]), x[k][2]), h = fmaxf(fmaxf(x[k][0], x[k][1]), x[k][2]);
        b.lo[k] = fminf(b.lo[k], l);
        b.hi[k] = fmaxf(b.hi[k], h);
        c[k] = 0.5f * l + 0.5f * h;
      }
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        float d2 = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) d2 = fmaf(x[k][v] - c[k], x[k][v] - c[k], d2);
        r2 = fmaxf(r2, d2);
      }
      const float m = fmaxf(fmaxf(fabsf(c[0]), fabsf(c[1])), fabsf(c[2]));
      sphere[f] = make_float4(c[0], c[1], c[2], fmaf(sqrtf(r2), 1.f + 1e-5f, 1e-6f * m));
    }
  }
  sb[t] = b;
  __syncthreads();
  const int blocks = (int)gridDim.x;
  // m nodes on this level within the block; their heap indices start at
  // blocks * m + blockIdx.x * m
  for (int m = per / 2; m >= 1; m >>= 1) {
    Box u;
    if (t < m) {
      const Box l = sb[2 * t], r = sb[2 * t + 1];
      store_node(node, (int64_t)blocks * m + (int64_t)blockIdx.x * m + t, l, r);
      u = join(l, r);
    }
    __syncthreads();
    if (t < m) sb[t] = u;
    __syncthreads();
  }
  if (blocks == 1) return;
  if (t == 0) {
    volatile float *o = block_box + 6 * (size_t)(blocks + blockIdx.x);   // heap slot of the root
    for (int k = 0; k < 3; ++k) { o[k] = sb[0].lo[k]; o[3 + k] = sb[0].hi[k]; }
    __threadfence();
    last = atomicAdd(&hdr->done, 1u) == (unsigned)blocks - 1u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int m = blocks / 2; m >= 1; m >>= 1) {
    for (int i = t; i < m; i += kBlock) {
      const volatile float *c = block_box + 6 * (size_t)(2 * (m + i));
      Box l, r;
      for (int k = 0; k < 3; ++k) {
        l.lo[k] = c[k]; l.hi[k] = c[3 + k]; r.lo[k] = c[6 + k]; r.hi[k] = c[9 + k];
      }
      store_node(node, m + i, l, r);
      const Box u = join(l, r);
      volatile float *o = block_box + 6 * (size_t)(m + i);
      for (int k = 0; k < 3; ++k) { o[k] = u.lo[k]; o[3 + k] = u.hi[k]; }
    }
    __threadfence_block();
    __syncthreads();
  }
}

__device__ __forceinline__ float box_dist2(V3<float> p, float lx, float ly, float lz, float hx,
                                           float hy, float hz) {
  const float dx = fmaxf(fmaxf(lx - p.x, p.x - hx), 0.f);
  const float dy = fmaxf(fmaxf(ly - p.y, p.y - hy), 0.f);
  const float dz = fmaxf(fmaxf(lz - p.z, p.z - hz), 0.f);
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Below this a square or a product may have lost bits to underflow: such a test is
// answered the safe way, or in FP64.
constexpr float kTiny = 1e-36f;

// Is the projected point left of the projected edge, taken upwards (from the
// end with y <= p.y to the other)?  0 when the edge does not pass p.y.  The
// sign is the edge's own direction.
__device__ __forceinline__ int edge_winding(V3<float> p, V3<float> a, V3<float> b) {
  const bool ua = a.y <= p.y, ub = b.y <= p.y;
  if (ua == ub) return 0;
  const V3<float> l = ua ? a : b, u = ua ? b : a;
  const int dir = ua ? 1 : -1;
  if (p.x < fminf(l.x, u.x)) return dir;
  if (p.x > fmaxf(l.x, u.x)) return 0;
  // left of the edge when (u.x - l.x)(p.y - l.y) > (p.x - l.x)(u.y - l.y);
  // FP32 decides where the products differ by more than their rounding
  const float f = (u.x - l.x) * (p.y - l.y), g = (p.x - l.x) * (u.y - l.y);
  if (fabsf(f - g) > fmaf(1e-6f, fabsf(f) + fabsf(g), kTiny)) return f > g ? dir : 0;
  const double s = ((double)u.x - l.x) * ((double)p.y - l.y) - ((double)p.x - l.x) * ((double)u.y - l.y);
  return s > 0.0 ? dir : 0;
}

// On which side of triangle (a, b, c) is p: the sign of ((b-a) x (c-a)).(a-p),
// positive behind it.
__device__ __forceinline__ float plane_side(V3<float> p, V3<float> a, V3<float> b, V3<float> c) {
  const V3<float> u = sub(b, a), v = sub(c, a), w = sub(a, p);
  const float x1 = u.y * v.z, x2 = u.z * v.y, y1 = u.z * v.x, y2 = u.x * v.z, z1 = u.x * v.y,
              z2 = u.y * v.x;
  const float s = (x1 - x2) * w.x + (y1 - y2) * w.y + (z1 - z2) * w.z;
  const float m = (fabsf(x1) + fabsf(x2)) * fabsf(w.x) + (fabsf(y1) + fabsf(y2)) * fabsf(w.y) +
                  (fabsf(z1) + fabsf(z2)) * fabsf(w.z);
  // (an underflowed x, y or z is off by a denormal, times w)
  if (fabsf(s) > fmaf(2e-6f, m, kTiny * (1.f + fabsf(w.x) + fabsf(w.y) + fabsf(w.z)))) return s;
  const V3<double> du = {(double)b.x - a.x, (double)b.y - a.y, (double)b.z - a.z};
  const V3<double> dv = {(double)c.x - a.x, (double)c.y - a.y, (double)c.z - a.z};
  const V3<double> dw = {(double)a.x - p.x, (double)a.y - p.y, (double)a.z - p.z};
  const double d = dot(cross(du, dv), dw);
  return d > 0.0 ? 1.f : (d < 0.0 ? -1.f : 0.f);
}

// Squared distance to the box of heap node i (a child of node i / 2).
__device__ __forceinline__ float node_dist2(V3<float> p, const float4 *__restrict__ node, unsigned i) {
  const float4 *nd = node + 3 * (size_t)(i >> 1);
  const float4 v = __ldg(nd + 1);
  if (i & 1u) {
    const float4 w = __ldg(nd + 2);
    return box_dist2(p, v.z, v.w, w.x, w.y, w.z, w.w);
  }
  const float4 u = __ldg(nd);
  return box_dist2(p, u.x, u.y, u.z, u.w, v.x, v.y);
}

// How far a box or a sphere may be and still hold a closer triangle than one at
// squared distance `best`: the triangle test's own rounding (slack, a few ulp of
// the coordinates) on top.
struct Reach {
  float r, r2;
};
__device__ __forceinline__ Reach reach_of(float best, float slack) {
  const float r = (sqrtf(best) + slack) * (1.f + 1e-6f);
  return {r, fminf(fmaf(r, r, kTiny), kFarDist2)};
}
// Can the triangle in sphere s be within reach of p?
__device__ __forceinline__ bool near_sphere(V3<float> p, const float4 &s, const Reach &reach) {
  const float dx = p.x - s.x, dy = p.y - s.y, dz = p.z - s.z, r = reach.r + s.w;
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= fmaf(r, r, kTiny);
}

// One point's search by `warps` warps, of which this is number `warp`: the tree
// is read as a 32-way one (nodes over 1024 triangles, over 32, the triangles), a
// lane per child, and the warps take the top nodes in turn.  `shared_best` (the
// bits of the smallest squared distance of all warps; or null for one warp)
// carries their results.  Every lane returns the smallest squared distance that
// it knows of, of triangles within `reach`.
__device__ float warp_search(V3<float> p, Reach reach, float slack, const float4 *__restrict__ tri,
                             const float4 *__restrict__ sphere, const float4 *__restrict__ node,
                             int leaves, unsigned warp, unsigned warps, unsigned *shared_best) {
  const unsigned lane = threadIdx.x & 31u;
  const unsigned groups = (unsigned)leaves / 8u;
  // top nodes: over 1024 triangles, or fewer when that leaves warps idle
  unsigned per = 32u;
  while (per > 1u && groups / per < 4u * warps) per >>= 1;
  const unsigned tops = (groups + per - 1u) / per;
  float best = INFINITY;
  for (unsigned t0 = 0; t0 < tops; t0 += 32u) {
    const unsigned t = t0 + lane;
    float dt = INFINITY;
    if (t < tops && t % warps == warp) dt = tops > 1u ? node_dist2(p, node, tops + t) : 0.f;
    unsigned tm = __ballot_sync(0xffffffffu, dt <= reach.r2);
    while (tm) {
      const unsigned ti = t0 + __ffs(tm) - 1;
      tm &= tm - 1;
      if (shared_best) {
        // read once for the whole warp: the other warps lower it meanwhile, and lanes
        // that saw different values would part before the next ballot
        unsigned bits = 0u;
        if (lane == 0u) bits = *(volatile unsigned *)shared_best;
        const float other = __uint_as_float(__shfl_sync(0xffffffffu, bits, 0));
        if (other < best) {
          best = other;
          const Reach closer = reach_of(best, slack);
          if (closer.r2 < reach.r2) reach = closer;
        }
      }
      const unsigned g = per * ti + lane;
      const float dg = lane < per && g < groups ? node_dist2(p, node, groups + g) : INFINITY;
      unsigned gm = __ballot_sync(0xffffffffu, dg <= reach.r2);
      while (gm) {
        const size_t f = (size_t)32 * (per * ti + __ffs(gm) - 1) + lane;
        gm &= gm - 1;
        float d = INFINITY;
        if (near_sphere(p, sphere[f], reach)) {
          const Tri q = load_tri(tri + 3 * f);
          d = tri_dist2(p, q.a, q.b, q.c);
        }
        // distances are not negative, so their bits order them (a NaN comes last)
        const unsigned m = __reduce_min_sync(0xffffffffu, __float_as_uint(d));
        if (__uint_as_float(m) < best) {
          best = __uint_as_float(m);
          if (shared_best && lane == 0) atomicMin(shared_best, m);
          const Reach closer = reach_of(best, slack);
          if (closer.r2 < reach.r2) reach = closer;
          gm &= __ballot_sync(0xffffffffu, dg <= reach.r2);
        }
      }
      tm &= __ballot_sync(0xffffffffu, dt <= reach.r2);
    }
  }
  return best;
}

// Coordinate k of p, and the ray's axes: it runs along axis A, the other two
// span the projection in an order that keeps its orientation.
template <int A>
__device__ __forceinline__ V3<float> along_z(V3<float> p) {
  if (A == 0) return {p.y, p.z, p.x};
  if (A == 1) return {p.z, p.x, p.y};
  return p;
}

// Winding number of the mesh about p: signed crossings of the ray from p along
// axis A, upwards (dir = 1) or downwards (dir = -1).
template <int A>
__device__ int ray_crossings(V3<float> p0, int dir, const float4 *__restrict__ tri,
                             const float4 *__restrict__ sphere, const float4 *__restrict__ node,
                             int leaves, int *stack) {
  const V3<float> p = along_z<A>(p0);
  int wind = 0, sp = 0, at = 1;
  auto meets = [&](V3<float> lo, V3<float> hi) {
    lo = along_z<A>(lo);
    hi = along_z<A>(hi);
    return p.x >= lo.x && p.x <= hi.x && p.y >= lo.y && p.y <= hi.y &&
           (dir > 0 ? p.z <= hi.z : p.z >= lo.z);
  };
  while (at) {
    while (at && at < leaves) {
      const float4 *nd = node + 3 * (size_t)at;
      const float4 u = __ldg(nd), v = __ldg(nd + 1), w = __ldg(nd + 2);
      const bool l = meets({u.x, u.y, u.z}, {u.w, v.x, v.y});
      const bool r = meets({v.z, v.w, w.x}, {w.y, w.z, w.w});
      if (l && r) stack[sp++] = 2 * at + 1;
      at = l ? 2 * at : (r ? 2 * at + 1 : (sp > 0 ? stack[--sp] : 0));
    }
    if (!at) break;
    const size_t f = (size_t)(at - leaves) * kLeaf;
    float4 c[kLeaf];
#pragma unroll
    for (int i = 0; i < kLeaf; ++i) c[i] = sphere[f + i];
#pragma unroll
    for (int i = 0; i < kLeaf; ++i) {
      const V3<float> m = along_z<A>({c[i].x, c[i].y, c[i].z});
      const float dx = p.x - m.x, dy = p.y - m.y;
      if (!(fmaf(dx, dx, dy * dy) <= fmaf(c[i].w, c[i].w, kTiny))) continue;
      const Tri q = load_tri(tri + 3 * (f + i));
      const V3<float> a = along_z<A>(q.a), b = along_z<A>(q.b), d = along_z<A>(q.c);
      const int wn = edge_winding(p, a, b) + edge_winding(p, b, d) + edge_winding(p, d, a);
      if (wn != 0) {
        // in front of p along the ray, and which way round
        const float side = plane_side(p, a, b, d);
        const bool above = wn > 0 ? side > 0.f : side < 0.f;
        const bool below = wn > 0 ? side < 0.f : side > 0.f;
        if (dir > 0 ? above : below) wind += dir * wn;
      }
    }
    at = sp > 0 ? stack[--sp] : 0;
  }
  return wind;
}

// Rounding of the distance test: coordinates of this size, a few ulp.
__device__ __forceinline__ float slack_of(V3<float> p, const MeshTreeHeader *__restrict__ hdr) {
  float scale = fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fabsf(p.z));
#pragma unroll
  for (int k = 0; k < 3; ++k)
    scale = fmaxf(scale, fmaxf(fabsf(unordered(hdr->neg_lo[k])), fabsf(unordered(hdr->hi[k]))));
  return 1e-6f * scale;
}

// Signed distance of every point: nearest-first descent for the distance, then
// the crossings of a ray for the sign.  A thread owns a point.  A point about as
// far from many triangles (the middle of a round body) would keep its thread
// descending long after the others are done, and neighbours of such a point are
// no better, so after a budget of leaves it is put on a list and searched by a
// block of its own (mesh_hard_kernel).
//
// Neighbouring threads take neighbouring points, so that a warp walks one part
// of the tree: explicit points in the Morton order of the build, grid nodes in
// bricks of 8 x 4 x 4 per block.
__global__ void __launch_bounds__(128) mesh_tree_kernel(const float4 *__restrict__ tri,
                                                        const float4 *__restrict__ sphere,
                                                        const float4 *__restrict__ node, int leaves,
                                                        const MeshTreeHeader *__restrict__ hdr,
                                                        const float4 *__restrict__ pts,
                                                        const unsigned *__restrict__ order, int64_t n,
                                                        float *__restrict__ out, const GridPts grid,
                                                        int budget, unsigned *hard_count,
                                                        int64_t *hard_list, unsigned hard_cap) {
  if (!mesh_tree_usable(hdr)) return;
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (!pts) {
    const int64_t N = grid.n, bx = (N + 7) / 8, by = (N + 3) / 4;
    const int64_t i = 8 * (blockIdx.x % bx) + (threadIdx.x & 7),
                  j = 4 * ((blockIdx.x / bx) % by) + ((threadIdx.x >> 3) & 3),
                  k = 4 * (blockIdx.x / (bx * by)) + (threadIdx.x >> 5);
    idx = i < N && j < N && k < N ? i + N * (j + N * k) : n;
  } else if (idx < n) {
    idx = order[idx];
  }
  V3<float> p = {0.f, 0.f, 0.f};
  if (idx < n) p = query_point(pts, grid, idx);
  const bool finite = fabsf(p.x) < INFINITY && fabsf(p.y) < INFINITY && fabsf(p.z) < INFINITY;
  const bool work = idx < n && finite;
  const float slack = slack_of(p, hdr);
  // the ray will run towards the nearest side of the mesh's box
  const float pc[3] = {p.x, p.y, p.z};
  float nearest = INFINITY;
  int axis = 2, dir = 1;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float up = unordered(hdr->hi[k]) - pc[k], down = pc[k] + unordered(hdr->neg_lo[k]);
    if (fminf(up, down) < nearest) {
      nearest = fminf(up, down);
      axis = k;
      dir = up <= down ? 1 : -1;
    }
  }

  int stack[kStack];
  float dist[kStack];
  int sp = 0, at = 1, left = budget;
  float best = kFarDist2;
  Reach reach = {INFINITY, kFarDist2};
  // the next box on the stack that may still hold a closer triangle (0: none)
  auto pop = [&]() -> int {
    while (sp > 0)
      if (dist[--sp] <= reach.r2) return stack[sp];
    return 0;
  };
  if (!work) at = 0;
  while (at) {
    while (at && at < leaves) {
      const float4 *nd = node + 3 * (size_t)at;
      const float4 u = __ldg(nd), v = __ldg(nd + 1), w = __ldg(nd + 2);
      const float dl = box_dist2(p, u.x, u.y, u.z, u.w, v.x, v.y);
      const float dr = box_dist2(p, v.z, v.w, w.x, w.y, w.z, w.w);
      const bool near_left = dl <= dr;
      const float dn = near_left ? dl : dr, df = near_left ? dr : dl;
      const int near = 2 * at + (near_left ? 0 : 1);
      if (df <= reach.r2) {
        stack[sp] = near ^ 1;
        dist[sp++] = df;
      }
      at = dn <= reach.r2 ? near : pop();
    }
    if (!at || left-- == 0) break;
    const size_t f = (size_t)(at - leaves) * kLeaf;
    float4 c[kLeaf];
#pragma unroll
    for (int i = 0; i < kLeaf; ++i) c[i] = sphere[f + i];
#pragma unroll 1
    for (int i = 0; i < kLeaf; ++i) {
      const float4 ci = i == 0 ? c[0] : i == 1 ? c[1] : i == 2 ? c[2] : c[3];
      if (!near_sphere(p, ci, reach)) continue;
      const Tri q = load_tri(tri + 3 * (f + i));
      const float d = tri_dist2(p, q.a, q.b, q.c);
      if (d < best) {
        best = d;
        reach = reach_of(best, slack);
      }
    }
    at = pop();
  }
  // a hard point goes on the list for mesh_hard_kernel, or, when that is full,
  // to this warp
  __syncwarp();
  bool hard = false;
  if (left < 0) {
    const unsigned at_list = atomicAdd(hard_count, 1u);
    if (at_list < hard_cap) hard_list[at_list] = idx;
    else hard = true;
  }
  unsigned todo = __ballot_sync(0xffffffffu, hard);
  while (todo) {
    const int q = __ffs(todo) - 1;
    todo &= todo - 1;
    const V3<float> pq = {__shfl_sync(0xffffffffu, p.x, q), __shfl_sync(0xffffffffu, p.y, q),
                          __shfl_sync(0xffffffffu, p.z, q)};
    const float sl = __shfl_sync(0xffffffffu, slack, q), bq = __shfl_sync(0xffffffffu, best, q);
    const float d = warp_search(pq, reach_of(bq, sl), sl, tri, sphere, node, leaves, 0u, 1u, nullptr);
    if ((int)(threadIdx.x & 31u) == q) best = fminf(best, d);
  }
  if (!work) {
    if (idx < n) out[idx] = sqrtf(kFarDist2);
    return;
  }

  // sign: any axis and direction give the same whole number
  const int wind = axis == 0   ? ray_crossings<0>(p, dir, tri, sphere, node, leaves, stack)
                   : axis == 1 ? ray_crossings<1>(p, dir, tri, sphere, node, leaves, stack)
                               : ray_crossings<2>(p, dir, tri, sphere, node, leaves, stack);
  const float d = sqrtf(best);
  out[idx] = wind >= 1 ? -d : d;
}

// The listed points: a warp each in turn, or, when they are few, a block each (its
// warps do not finish together, and half of them would wait at the block's
// barriers).  out holds the sign and an upper bound of the distance, which stays
// where the search finds nothing (no triangle whose distance FP32 can hold).
__global__ void __launch_bounds__(32 * kHardWarps) mesh_hard_kernel(
    const float4 *__restrict__ tri, const float4 *__restrict__ sphere, const float4 *__restrict__ node,
    int leaves, const MeshTreeHeader *__restrict__ hdr, const float4 *__restrict__ pts,
    float *__restrict__ out, const GridPts grid, const unsigned *__restrict__ hard_count,
    const int64_t *__restrict__ hard_list, unsigned hard_cap) {
  __shared__ unsigned best_bits;
  const unsigned count = min(*hard_count, hard_cap);
  if (count > 10u * gridDim.x) {
    for (unsigned i = blockIdx.x * kHardWarps + (threadIdx.x >> 5); i < count;
         i += gridDim.x * kHardWarps) {
      const int64_t idx = hard_list[i];
      const V3<float> p = query_point(pts, grid, idx);
      const float slack = slack_of(p, hdr), d = out[idx];
      const float best = warp_search(p, reach_of(d * d * (1.f + 1e-6f), slack), slack, tri, sphere, node,
                                     leaves, 0u, 1u, nullptr);
      if ((threadIdx.x & 31u) == 0u) out[idx] = copysignf(fminf(sqrtf(best), fabsf(d)), d);
    }
    return;
  }
  for (unsigned i = blockIdx.x; i < count; i += gridDim.x) {
    const int64_t idx = hard_list[i];
    const V3<float> p = query_point(pts, grid, idx);
    const float slack = slack_of(p, hdr), d = out[idx];
    if (threadIdx.x == 0) best_bits = 0x7f800000u;
    __syncthreads();
    // (the root rounds: a little more than its square)
    warp_search(p, reach_of(d * d * (1.f + 1e-6f), slack), slack, tri, sphere, node, leaves,
                threadIdx.x >> 5, kHardWarps, &best_bits);
    __syncthreads();
    if (threadIdx.x == 0)
      out[idx] = copysignf(fminf(sqrtf(__uint_as_float(best_bits)), fabsf(d)), d);
    __syncthreads();
  }
}

}  // namespace

size_t mesh_tree_bytes(int64_t n_faces, int64_t n_points, int64_t n_nodes) {
  return tree_mem(n_faces, n_points, n_nodes).total;
}

cudaError_t launch_mesh_tree(const float *verts, int64_t n_verts, const int32_t *faces,
                             int64_t n_faces, const float4 *pts, int64_t n, float *out,
                             const GridPts &grid, void *mem, cudaStream_t s) {
  const TreeMem m = tree_mem(n_faces, pts ? n : 0, pts ? 0 : n);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int hard_blocks = kHardPerSm * sms;
  char *base = static_cast<char *>(mem);
  MeshTreeHeader *hdr = reinterpret_cast<MeshTreeHeader *>(base + m.header);
  unsigned *hist = reinterpret_cast<unsigned *>(base + m.hist);
  unsigned *hard_count = reinterpret_cast<unsigned *>(base + m.hard_count);
  int64_t *hard = reinterpret_cast<int64_t *>(base + m.hard);
  unsigned *phist = reinterpret_cast<unsigned *>(base + m.phist);
  uint2 *key = reinterpret_cast<uint2 *>(base + m.key);
  uint2 *pkey = reinterpret_cast<uint2 *>(base + m.pkey);
  unsigned *order = reinterpret_cast<unsigned *>(base + m.order);
  float4 *tri = reinterpret_cast<float4 *>(base + m.tri);
  float4 *sphere = reinterpret_cast<float4 *>(base + m.sphere);
  float4 *node = reinterpret_cast<float4 *>(base + m.node);
  float *block_box = reinterpret_cast<float *>(base + m.block_box);
  const int cells = 1 << (3 * m.bits), pcells = 1 << (3 * kPointBits);
  e = cudaMemsetAsync(base + m.header, 0, m.key - m.header, s);
  if (e != cudaSuccess) return e;
  unsigned fb = (unsigned)((n_faces + kBlock - 1) / kBlock);
  tree_bounds_kernel<<<fb < 1024 ? fb : 1024, kBlock, 0, s>>>(verts, n_verts, faces, n_faces, hdr);
  for (int64_t c0 = 0; c0 < n; c0 += m.chunk) {
    // the faces' part of the sort belongs to the first chunk of points
    const int64_t k = pts ? (n - c0 < m.chunk ? n - c0 : m.chunk) : 0;
    if (c0 > 0) {
      fb = 0;
      e = cudaMemsetAsync(base + m.hard_count, 0, m.phist - m.hard_count + sizeof(unsigned) * pcells, s);
      if (e != cudaSuccess) return e;
    }
    const unsigned blocks = fb + (unsigned)((k + kBlock - 1) / kBlock);
    const float4 *cp = pts ? pts + c0 : nullptr;
    tree_cell_kernel<<<blocks, kBlock, 0, s>>>(verts, n_verts, faces, n_faces, m.bits, fb, cp, k, hdr,
                                              hist, key, phist, pkey);
    if (fb > 0) tree_scan_kernel<<<pts ? 2 : 1, 1024, 0, s>>>(hdr, hist, cells, phist, pcells);
    else tree_scan_kernel<<<1, 1024, 0, s>>>(hdr, phist, pcells, nullptr, 0);
    tree_scatter_kernel<<<blocks, kBlock, 0, s>>>(verts, n_verts, faces, n_faces, fb, k, hdr, hist, key,
                                                 phist, pkey, tri, order);
    if (fb > 0) {
      const int64_t bb = m.leaves < kBlock ? 1 : m.leaves / kBlock;
      tree_box_kernel<<<(unsigned)bb, kBlock, 0, s>>>(tri, sphere, node, (int)m.leaves, block_box,
                                                      hdr);
    }
    int64_t qb = (k + 127) / 128, count = k;
    if (!pts) {
      const int64_t N = grid.n;
      qb = ((N + 7) / 8) * ((N + 3) / 4) * ((N + 3) / 4);
      count = n;
    }
    mesh_tree_kernel<<<(unsigned)qb, 128, 0, s>>>(tri, sphere, node, (int)m.leaves, hdr, cp, order,
                                                 count, out + c0, grid,
                                                 n <= kFewPerBlock * (int64_t)hard_blocks ? kLeafBudgetFew : kLeafBudget,
                                                 hard_count, hard, m.hard_cap);
    mesh_hard_kernel<<<hard_blocks, 32 * kHardWarps, 0, s>>>(tri, sphere, node, (int)m.leaves, hdr, cp,
                                                            out + c0, grid, hard_count, hard, m.hard_cap);
    if (!pts) break;
  }
  return cudaGetLastError();
}

}  // namespace nsdf
