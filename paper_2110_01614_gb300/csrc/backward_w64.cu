// Backward of the network query for width 64 with two or three hidden layers
// (FP32, CUDA cores): the computation of backward.cu, blocked in registers.
//
// The primal and the tangent value of an element travel as one f32x2 pair
// (x, xd), so each product of the forward pass and of the reverse pass is one
// paired FMA with the weight in both lanes, and the weight gradient
// sum_p zb x + zdb xd is one paired FMA whose lanes are added at the end.  A
// CTA of 256 threads takes a tile of 64 points; a thread owns 4 points x 4
// columns of every layer (its slopes and tangents stay in registers from the
// forward to the reverse pass) and 4 x 4 elements of every weight gradient,
// which are summed over the tile in registers and added once per tile to the
// CTA's totals in shared memory.  Per k step a thread reads 16 bytes of weights
// and 32 bytes of pairs for 16 paired FMAs.
//
// Layouts in shared memory: weights [n][k] with the 16-byte chunk k / 4 of row n
// at chunk (k / 4) ^ (n / 4 mod 8), so that the forward product (one chunk of
// eight threads' rows) and the reverse one (eight chunks of a row) both read
// eight different banks; pairs [column][point] with rows of 132 floats, so that
// neighbouring rows lie in different banks.  Lanes that differ in bit 1 share
// their columns, lanes that differ in bit 0 their points: 16-byte shared loads
// then merge into two wavefronts instead of four.
//
// Bound: the FP32 pipe (50 K FMA a point with both streams: 0.33 ms for 250,000
// points at its rate).  Measured, 250,000 points of 3-64-64-64-1 with weight
// gradients: general kernel 3.45 ms, this one 0.66 ms (0.61 with the hardware's
// approximate exp, log and quotient, whose error grows with 1 / beta; 0.76 with IEEE
// quotients).  Eight point pairs and four columns per warp, whose shared loads take ten
// wavefronts a k step where this mapping takes six, cost 3%.

#include "backward.cuh"
#include "f32x2.cuh"

namespace nsdf {
namespace {

constexpr int kW = 64;
constexpr int kP = 64;                    // points per tile
constexpr int kThreads = 256;
constexpr int kARow = 2 * kP + 4;         // floats per row of pairs
constexpr int kShort = kW - 3;            // outputs of the layer feeding a skip
constexpr float kInvSqrt2 = 0.70710678118654752f;

// Shared-memory map, in floats.
template <int L>
struct Map {
  static constexpr int w = 0;                              // [L-1][kW][kW], swizzled
  static constexpr int a = w + (L - 1) * kW * kW;       // [L-1][kW][kARow]: layer inputs
  static constexpr int zb = a + (L - 1) * kW * kARow;      // [kW][kARow]
  static constexpr int gw = zb + kW * kARow;               // [L-1][4][kThreads] float4
  static constexpr int pv = gw + (L - 1) * 16 * kThreads;  // [3][kARow]: pairs (p, v)
  static constexpr int av = pv + 3 * kARow;                // [kP]
  static constexpr int w0 = av + kP;                       // [kW][4]
  static constexpr int bias = w0 + 4 * kW;                 // [L][kW]
  static constexpr int wout = bias + L * kW;               // [kW]
  static constexpr int dir = wout + kW;                    // [kP][4]: the skip's direct path
  static constexpr int red = dir + 4 * kP;                 // [16][kW]
  static constexpr int total = red + 16 * kW;
};

// As softplus_and_slope, with the two quotients by a residual step each (Newton's
// method: 1 + e lies in [1, 2], and inv_beta is beta's reciprocal).
__device__ __forceinline__ void softplus_and_slope_w64(float z, float beta, float inv_beta, float &h,
                                                       float &s) {
  const float e = expf(-beta * fabsf(z)), l = log1pf(e), d = 1.0f + e;
  const float q = l * inv_beta;
  h = fmaxf(z, 0.0f) + fmaf(fmaf(-q, beta, l), inv_beta, q);
  const float r = __fdividef(1.0f, d), inv = fmaf(fmaf(-d, r, 1.0f), r, r);
  s = (z >= 0.0f) ? inv : e * inv;
}

// Float offset of 16-byte chunk q of weight row n (rows of all layers in turn).
__device__ __forceinline__ int swizzled(int n, int q) { return n * kW + ((q ^ ((n >> 2) & 7)) << 2); }
__device__ __forceinline__ float2 lo(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi(const float4 &v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float el(const float4 &v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

template <int L>
__global__ void __launch_bounds__(kThreads, 1)
    backward_w64_kernel(const __grid_constant__ BwdParams prm) {
  using M = Map<L>;
  extern __shared__ float4 smem4[];
  float *sm = reinterpret_cast<float *>(smem4);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // forward / reverse: points 2 pg, 2 pg + 1, 32 + 2 pg, 33 + 2 pg; columns 4 cg .. 4 cg + 3
  const int pg = ((lane >> 1) & 1) + ((lane >> 2) & 2) + 4 * (warp & 3);
  const int cg = (lane & 1) + ((lane >> 1) & 2) + ((lane >> 2) & 4) + 8 * (warp >> 2);
  // weight gradients: rows pg + 16 i, columns cg + 16 j
  const int skip = prm.skip;
  const float beta = prm.beta, inv_beta = 1.0f / prm.beta;
  const bool weights = prm.g_partial != nullptr;

  for (int i = tid; i < (L - 1) * kW * kW; i += kThreads)
    sm[M::w + swizzled(i / kW, (i % kW) >> 2) + (i & 3)] = prm.bwd[i];
  for (int i = tid; i < kW * 3; i += kThreads) sm[M::w0 + (i / 3) * 4 + i % 3] = prm.w0[i];
  for (int i = tid; i < L * kW; i += kThreads) sm[M::bias + i] = prm.bias[i];
  for (int i = tid; i < kW; i += kThreads) sm[M::wout + i] = prm.wout[i];
  float4 *gw = reinterpret_cast<float4 *>(sm + M::gw);
  for (int i = 0; i < (L - 1) * 4; ++i) gw[i * kThreads + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
  // totals of this thread: w_out columns (over its points), b_out, and for row
  // tid / 4 over points 16 (tid % 4) .. + 15 the biases and W_0
  float t_wout[4] = {0.f, 0.f, 0.f, 0.f}, t_a = 0.f, t_b[L], t_w0[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int l = 0; l < L; ++l) t_b[l] = 0.f;
  const int rc = tid >> 2, rp = 16 * (tid & 3);
  float *zb = sm + M::zb;

  const int64_t ntiles = (prm.n + kP - 1) / kP;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t base = tile * kP;
    if (tid < kP) {
      const int64_t i = base + tid;
      float4 p = make_float4(0.f, 0.f, 0.f, 0.f), v = p;
      float a = 0.f;
      if (i < prm.n) {
        p = prm.pts[i];
        a = prm.a[i];
        if (prm.v) v = prm.v[i];
      }
      float2 *pv = reinterpret_cast<float2 *>(sm + M::pv) + tid;
      pv[0] = make_float2(p.x, v.x);
      pv[kARow / 2] = make_float2(p.y, v.y);
      pv[kARow] = make_float2(p.z, v.z);
      sm[M::av + tid] = a;
      t_a += a;
      reinterpret_cast<float4 *>(sm + M::dir)[tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();

    // ---- forward, (primal, tangent) pairs ----
    float2 acc[4][4];                    // [column][point]
    float s[L][4][4], zd[L][4][4];
#pragma unroll
    for (int l = 0; l < L; ++l) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float b = sm[M::bias + l * kW + 4 * cg + j];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[j][i] = make_float2(b, 0.f);
      }
      if (l == 0) {
        float4 w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4 *>(sm + M::w0 + 4 * (4 * cg + j));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float4 xa = *reinterpret_cast<const float4 *>(sm + M::pv + k * kARow + 4 * pg);
          const float4 xb = *reinterpret_cast<const float4 *>(sm + M::pv + k * kARow + 4 * pg + 64);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 ww = f2_splat(el(w[j], k));
            acc[j][0] = f2_fma(ww, lo(xa), acc[j][0]);
            acc[j][1] = f2_fma(ww, hi(xa), acc[j][1]);
            acc[j][2] = f2_fma(ww, lo(xb), acc[j][2]);
            acc[j][3] = f2_fma(ww, hi(xb), acc[j][3]);
          }
        }
      } else {
        const float *wl = sm + M::w + (l - 1) * kW * kW;
        const float *xl = sm + M::a + (l - 1) * kW * kARow + 4 * pg;
#pragma unroll 2
        for (int k = 0; k < kW; k += 4) {
          float4 w[4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            w[j] = *reinterpret_cast<const float4 *>(wl + swizzled(4 * cg + j, k >> 2));
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 xa = *reinterpret_cast<const float4 *>(xl + (k + q) * kARow);
            const float4 xb = *reinterpret_cast<const float4 *>(xl + (k + q) * kARow + 64);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float2 ww = f2_splat(el(w[j], q));
              acc[j][0] = f2_fma(ww, lo(xa), acc[j][0]);
              acc[j][1] = f2_fma(ww, hi(xa), acc[j][1]);
              acc[j][2] = f2_fma(ww, lo(xb), acc[j][2]);
              acc[j][3] = f2_fma(ww, hi(xb), acc[j][3]);
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 4 * cg + j;
        float2 x[4];
        float wsum = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float h;
          softplus_and_slope_w64(acc[j][i].x, beta, inv_beta, h, s[l][j][i]);
          zd[l][j][i] = acc[j][i].y;
          x[i] = make_float2(h, s[l][j][i] * acc[j][i].y);
          if (l == L - 1) {
            const int p = 2 * pg + (i & 1) + 16 * (i & 2);
            wsum += fmaf(sm[M::av + p], h, x[i].y);
          }
        }
        if (l == L - 1) {
          t_wout[j] += wsum;
        } else {
          if (l + 1 == skip) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (c >= kShort) {          // the input p (and its tangent v) joins here
                const int p = 2 * pg + (i & 1) + 16 * (i & 2);
                x[i] = *reinterpret_cast<const float2 *>(sm + M::pv + (c - kShort) * kARow + 2 * p);
              }
              x[i] = f2_mul(x[i], f2_splat(kInvSqrt2));
            }
          }
          float *o = sm + M::a + (l * kW + c) * kARow + 4 * pg;
          *reinterpret_cast<float4 *>(o) = make_float4(x[0].x, x[0].y, x[1].x, x[1].y);
          *reinterpret_cast<float4 *>(o + 64) = make_float4(x[2].x, x[2].y, x[3].x, x[3].y);
        }
      }
      if (l < L - 1) __syncthreads();
    }

    // ---- reverse over both streams: acc = (hb, hdb) of the layer's outputs ----
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float w = sm[M::wout + 4 * cg + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        acc[j][i] = make_float2(sm[M::av + 2 * pg + (i & 1) + 16 * (i & 2)] * w, w);
    }
#pragma unroll
    for (int l = L - 1; l >= 0; --l) {
      const int outl = prm.out[l];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 4 * cg + j;
        float2 z[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float sl = s[l][j][i], hdb = acc[j][i].y;
          z[i] = make_float2(fmaf(sl, acc[j][i].x, zd[l][j][i] * hdb * beta * sl * (1.0f - sl)), sl * hdb);
          if (c >= outl) z[i] = make_float2(0.f, 0.f);
        }
        float *o = zb + c * kARow + 4 * pg;
        *reinterpret_cast<float4 *>(o) = make_float4(z[0].x, z[0].y, z[1].x, z[1].y);
        *reinterpret_cast<float4 *>(o + 64) = make_float4(z[2].x, z[2].y, z[3].x, z[3].y);
      }
      __syncthreads();
      if (weights) {
        // bias of row rc (and W_0): points rp .. rp + 15
        float b = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f;
#pragma unroll 4
        for (int p = 0; p < 16; p += 2) {
          const float4 z = *reinterpret_cast<const float4 *>(zb + rc * kARow + 2 * (rp + p));
          b += z.x + z.z;
          if (l == 0) {
            const float *x = sm + M::pv + 2 * (rp + p);
            const float4 x0 = *reinterpret_cast<const float4 *>(x);
            const float4 x1 = *reinterpret_cast<const float4 *>(x + kARow);
            const float4 x2 = *reinterpret_cast<const float4 *>(x + 2 * kARow);
            g0 += fmaf(z.x, x0.x, z.y * x0.y) + fmaf(z.z, x0.z, z.w * x0.w);
            g1 += fmaf(z.x, x1.x, z.y * x1.y) + fmaf(z.z, x1.z, z.w * x1.w);
            g2 += fmaf(z.x, x2.x, z.y * x2.y) + fmaf(z.z, x2.z, z.w * x2.w);
          }
        }
        t_b[l] += b;
        if (l == 0) { t_w0[0] += g0; t_w0[1] += g1; t_w0[2] += g2; }
      }
      if (l == 0) {
        if (prm.g_pts) {
          // dL/dp = W_0^T zb (+ the skip's direct path); point tid / 4, 16 rows per lane
          float g0 = 0.f, g1 = 0.f, g2 = 0.f;
          const int p = tid >> 2;
          for (int c = rp; c < rp + 16; ++c) {
            const float z = zb[c * kARow + 2 * p];
            const float4 w = *reinterpret_cast<const float4 *>(sm + M::w0 + 4 * c);
            g0 = fmaf(z, w.x, g0); g1 = fmaf(z, w.y, g1); g2 = fmaf(z, w.z, g2);
          }
#pragma unroll
          for (int o = 1; o < 4; o <<= 1) {
            g0 += __shfl_xor_sync(0xffffffffu, g0, o);
            g1 += __shfl_xor_sync(0xffffffffu, g1, o);
            g2 += __shfl_xor_sync(0xffffffffu, g2, o);
          }
          const float4 d = reinterpret_cast<const float4 *>(sm + M::dir)[p];
          if ((tid & 3) == 0 && base + p < prm.n)
            prm.g_pts[base + p] = make_float4(g0 + d.x, g1 + d.y, g2 + d.z, 0.f);
        }
        break;
      }
      const float *xl = sm + M::a + (l - 1) * kW * kARow;
      if (weights) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int p = 0; p < kP; p += 2) {
          float4 z[4], x[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            z[i] = *reinterpret_cast<const float4 *>(zb + (pg + 16 * i) * kARow + 2 * p);
            x[i] = *reinterpret_cast<const float4 *>(xl + (cg + 16 * i) * kARow + 2 * p);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              acc[i][j] = f2_fma(lo(z[i]), lo(x[j]), acc[i][j]);
              acc[i][j] = f2_fma(hi(z[i]), hi(x[j]), acc[i][j]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float4 *g = gw + ((l - 1) * 4 + i) * kThreads + tid;
          float4 t = *g;
          t.x += acc[i][0].x + acc[i][0].y;
          t.y += acc[i][1].x + acc[i][1].y;
          t.z += acc[i][2].x + acc[i][2].y;
          t.w += acc[i][3].x + acc[i][3].y;
          *g = t;
        }
      }
      // (hb, hdb) of layer l - 1: W_l^T (zb, zdb)
      const float *wl = sm + M::w + (l - 1) * kW * kW;
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[j][i] = make_float2(0.f, 0.f);
#pragma unroll 4
      for (int c = 0; c < kW; ++c) {
        const float4 w = *reinterpret_cast<const float4 *>(wl + swizzled(c, cg));
        const float4 za = *reinterpret_cast<const float4 *>(zb + c * kARow + 4 * pg);
        const float4 zc = *reinterpret_cast<const float4 *>(zb + c * kARow + 4 * pg + 64);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 ww = f2_splat(el(w, j));
          acc[j][0] = f2_fma(ww, lo(za), acc[j][0]);
          acc[j][1] = f2_fma(ww, hi(za), acc[j][1]);
          acc[j][2] = f2_fma(ww, lo(zc), acc[j][2]);
          acc[j][3] = f2_fma(ww, hi(zc), acc[j][3]);
        }
      }
      if (l == skip) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int k = 4 * cg + j;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            acc[j][i] = f2_mul(acc[j][i], f2_splat(kInvSqrt2));
            if (k >= kShort) {            // straight to the input
              sm[M::dir + 4 * (2 * pg + (i & 1) + 16 * (i & 2)) + k - kShort] = acc[j][i].x;
              acc[j][i] = make_float2(0.f, 0.f);
            }
          }
        }
      }
      __syncthreads();                    // zb is rewritten for layer l - 1
    }
    __syncthreads();                      // the next tile's inputs replace pv, av, zb
  }
  if (!weights) return;

  // ---- this CTA's partial sums, in blob layout ----
  float *dst = prm.g_partial + (size_t)blockIdx.x * prm.n_params;
#pragma unroll
  for (int l = 1; l < L; ++l)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = pg + 16 * i;
      const float4 g = gw[((l - 1) * 4 + i) * kThreads + tid];
      if (c < prm.out[l]) {
        float *o = dst + prm.woff[l] + (int64_t)c * kW + cg;
        o[0] = g.x; o[16] = g.y; o[32] = g.z; o[48] = g.w;
      }
    }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
#pragma unroll
    for (int l = 0; l < L; ++l) t_b[l] += __shfl_xor_sync(0xffffffffu, t_b[l], o);
#pragma unroll
    for (int k = 0; k < 3; ++k) t_w0[k] += __shfl_xor_sync(0xffffffffu, t_w0[k], o);
  }
  if ((tid & 3) == 0) {
#pragma unroll
    for (int l = 0; l < L; ++l)
      if (rc < prm.out[l]) dst[prm.boff[l] + rc] = t_b[l];
    if (rc < prm.out[0])
      for (int k = 0; k < 3; ++k) dst[prm.woff[0] + 3 * rc + k] = t_w0[k];
  }
  // w_out over the 16 point groups, b_out over the 64 points (a tree: one chain of 64
  // sums loses the small ones)
#pragma unroll
  for (int j = 0; j < 4; ++j) sm[M::red + pg * kW + 4 * cg + j] = t_wout[j];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t_a += __shfl_xor_sync(0xffffffffu, t_a, o);
  if (lane == 0 && warp < kP / 32) sm[M::av + warp] = t_a;
  __syncthreads();
  if (tid < kW) {
    float t = 0.f;
    for (int g = 0; g < 16; ++g) t += sm[M::red + g * kW + tid];
    dst[prm.woff[L] + tid] = t;
  }
  if (tid == 0) dst[prm.boff[L]] = sm[M::av] + sm[M::av + 1];
}

template <int L>
cudaError_t launch_t(const BwdParams &p, int grid, cudaStream_t s) {
  constexpr int smem = Map<L>::total * (int)sizeof(float);
  static_assert(smem <= 232448, "shared memory");
  cudaError_t e = cudaFuncSetAttribute(backward_w64_kernel<L>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  backward_w64_kernel<L><<<grid, kThreads, smem, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

bool backward_w64_supported(int width, int n_hidden) {
  return width == kW && (n_hidden == 2 || n_hidden == 3);
}

cudaError_t launch_backward_w64(const BwdParams &p, int grid, cudaStream_t s) {
  return p.L == 2 ? launch_t<2>(p, grid, s) : launch_t<3>(p, grid, s);
}

}  // namespace nsdf
