// FP32 CUDA-core form of the fused collision query.
//
// A persistent CTA (64 to 512 threads, by the width and the tile shape) walks tiles of
// P points.  For each tile it runs, without leaving the SM:
//   * L0 (K = 3) on CUDA cores,
//   * the hidden layers z_l = W_l x_l + b_l, h_l = softplus_beta(z_l) (Eq. 1)
//     as register-blocked products against weight panels staged in shared
//     memory with cp.async,
//   * the output unit f = w_out . h + b_out,
//   * the Jacobian-transpose chain of Sec. 3.2: delta_l = sigmoid(beta z_l) *
//     g_l, g_{l-1} = W_l^T delta_l, down to grad f = W_0^T delta_0 (plus the
//     skip connection's direct term),
//   * Eq. 2 (normalise), the collision test f < eps and the contact point of
//     Eq. 3, with the optional rigid transform of Sec. 4.2.
// The paper's own networks (Sec. 4.3: a Fourier-feature layer, then ReLU
// layers) run through the same loop: gamma(p) = [sin(2 pi B p),
// cos(2 pi B p)] is written as the input tile of L0, which becomes a
// width x width panel product; the ReLU slope is the 0/1 step; and the
// reverse chain ends with g_gamma = W_0^T delta_0 folded into grad f through
// the feature Jacobian.
// sigmoid(beta z_l) of every hidden layer is parked in a per-CTA scratch
// slab between the forward and the reverse pass; it is written and read by
// the same thread in a lane-contiguous order (coalesced, L2-resident).
//
// Products.  A thread owns 8 points x TC columns (TC = 8 from width 256 on, 4
// below); a warp covers 32 points x 8 TC columns, a CTA PW x CW warps.  The
// activation tile is stored [column][point], so a thread reads its points as
// natural pairs and multiplies each pair by a weight in both lanes of one
// f32x2 FMA: per k step 2 x 16 bytes of points and TC / 4 x 16 bytes of weights
// feed 4 TC paired FMAs.  With the scalar form (a warp on one group of 8
// points, weights read as single words) the issue slots and the shared-memory
// reads bounded the kernel at 0.54 of the FMA rate; here the FP32 pipe is busy
// 0.7 of the time (a paired FMA beside the moves that double a weight runs at
// 0.75-0.88 of the pipe in a probe; scalar FMAs in this layout measure 3-9%
// slower).  Measured, before -> now: 131,077 points of 3-512x8-1 22.9 -> 16.9 ms,
// 300,000 of the 8 x 256 Fourier-feature network 16.8 -> 11.1 ms, 1,048,576 of
// 3-64x3-1 1.23 -> 0.77 ms, 1,000 points of 3-512x8-1 0.85 -> 0.66 ms.
// Each accumulator is the same chain of FMAs over k, so z, the activations and
// the slopes keep their bits.  A layer's output replaces its input in place
// once every warp has read it, which leaves room for tiles of 64 points at
// width 512 (half the weight traffic of 32); the weight panels of all layers
// are one stream of chunks through a cp.async ring that runs ahead across the
// layers' epilogues, with one barrier per chunk.
//
// The small shape (PT = 4, half the warps and half the points per tile) is for
// launches whose small tiles all fit on the GPU at once, where a larger tile would
// leave SMs idle, for grouped launches of small bodies, and for calls whose scratch
// holds too few of the large tile's slabs (the rules are in query_fp32.cu).

#pragma once

#include "f32x2.cuh"
#include "ff_phase.cuh"
#include "nsdf_internal.h"

namespace nsdf {
namespace {

constexpr float kInvSqrt2 = 0.70710678118654752f;

template <int W, int PT_ = 8>
struct Cfg {
  static constexpr int TP = 8;                          // points per thread
  static constexpr int TC = W >= 256 ? 8 : 4;           // columns per thread
  static constexpr int CW = W / (8 * TC);               // warps across the columns
  static constexpr int PW = (W <= 64 ? 4 : 2) / (PT_ == 4 ? 2 : 1);   // warps across the points
  static constexpr int THREADS = 32 * CW * PW;
  static constexpr int P = 32 * PW;                     // points per tile
  static constexpr int XS = P + 4;                      // floats per activation row
  // panel rows per chunk (at width 512 chunks of 8 rows cost 5-12% more: each chunk
  // has its barrier and its copies' addresses)
  static constexpr int KC = W == 512 ? 16 : (4096 / W > W ? W : 4096 / W);
  static constexpr int NCHUNK = W / KC;
  static constexpr int NS = 2;                          // ring slots
  // CTAs per SM that the registers are budgeted for
  static constexpr int MIN_CTAS = THREADS >= 512 ? 1 : (W >= 128 ? 512 / THREADS : 768 / THREADS);
  static_assert(W % (8 * TC) == 0 && W % KC == 0 && P <= THREADS, "shape");
  // shared memory carve-up (floats)
  static constexpr int X_OFF = 0;
  static constexpr int M_OFF = X_OFF + XS * W;
  static constexpr int PS_OFF = M_OFF + NS * KC * W;         // float4 [P]
  static constexpr int RED_OFF = PS_OFF + 4 * P;             // [CW][P][4]
  static constexpr int DIR_OFF = RED_OFF + CW * P * 4;       // [P][4]
  static constexpr int SMEM_FLOATS = DIR_OFF + 4 * P;
  static constexpr size_t SMEM_BYTES = sizeof(float) * SMEM_FLOATS;
  static_assert(SMEM_BYTES <= 232448, "shared memory");
};

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

// softplus_beta(z) = max(z,0) + log1p(u)/beta and its derivative
// sigmoid(beta z), both from the same u = exp(-beta|z|) in (0, 1].  The
// hardware approximations suffice for the FP32 form: log(1 + u) on [1, 2]
// carries an absolute error of about 2^-21 and forming 1 + u at most ulp(1)/2,
// both divided by beta (1e-9 for beta = 100); exp and the reciprocal err by
// a few ulp relative, which moves u and the slope by about 1e-6 relative.
__device__ __forceinline__ void softplus_and_slope(float z, float beta, float inv_beta, float &h,
                                                   float &s) {
  const float u = __expf(-beta * fabsf(z));
  const float one_u = 1.0f + u;
  h = fmaf(__logf(one_u), inv_beta, fmaxf(z, 0.0f));
  const float inv = __fdividef(1.0f, one_u);
  s = (z >= 0.0f) ? inv : u * inv;
}

// The activation (softplus_beta or ReLU) and its slope.
__device__ __forceinline__ void act_and_slope(float z, float beta, float inv_beta, int relu, float &h,
                                              float &s) {
  if (relu) {
    h = fmaxf(z, 0.0f);
    s = z > 0.0f ? 1.0f : 0.0f;   // no gradient through a ReLU that outputs 0
  } else {
    softplus_and_slope(z, beta, inv_beta, h, s);
  }
}

__device__ __forceinline__ float el4(const float4 &v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

// FF: the network has the Fourier-feature input layer (compiled separately,
// so that networks without it keep the registers, hence the occupancy, of a
// kernel without that code).
template <int W, int PT_ = 8, bool FF = false>
__global__ void __launch_bounds__(Cfg<W, PT_>::THREADS, Cfg<W, PT_>::MIN_CTAS)
    query_fp32_kernel(const __grid_constant__ QueryParams prm) {
  using C = Cfg<W, PT_>;
  extern __shared__ float4 smem4[];
  float *smem = reinterpret_cast<float *>(smem4);
  float *X = smem + C::X_OFF;
  float *Ms = smem + C::M_OFF;
  float4 *Ps = reinterpret_cast<float4 *>(smem + C::PS_OFF);
  float *red = smem + C::RED_OFF;
  float *dir = smem + C::DIR_OFF;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cw = warp % C::CW, pw = warp / C::CW;
  // this thread's points: pb .. pb + 3 and pb + 16 .. pb + 19; columns cb .. cb + 3
  // (and cb + 32 .. cb + 35 when TC = 8)
  // (lanes that differ in bit 0 share their points, lanes that differ in bit 1
  // their columns: 16-byte shared loads then merge, two wavefronts instead of four)
  const int lp = ((lane >> 1) & 1) | ((lane >> 2) & 2),
            lc = (lane & 1) | ((lane >> 1) & 2) | ((lane >> 2) & 4);
  const int pb = 32 * pw + 4 * lp, cb = cw * 8 * C::TC + 4 * lc;
  auto point = [&](int i) { return pb + (i < 4 ? i : 12 + i); };
  auto column = [&](int j) { return cb + (j < 4 ? j : 28 + j); };
  const int L = prm.n_hidden;
  const int skip = prm.skip;
  const int nshort = W - 3;   // outputs of the layer feeding the skip
  const float beta = prm.beta;
  const float inv_beta = 1.0f / prm.beta;
  const bool grouped = prm.g_nets > 0;
  const int64_t ntiles = grouped ? (int64_t)prm.g_tile_start[prm.g_nets] : (prm.n + C::P - 1) / C::P;
  // per-CTA slope slab: [L-1][TC][2][THREADS] float4
  float4 *slab = reinterpret_cast<float4 *>(prm.scratch) +
                 (size_t)blockIdx.x * (size_t)(L > 1 ? L - 1 : 1) * (C::P * W / 4);
  auto slot = [&](int l, int j, int half) -> float4 * {
    return slab + ((size_t)(l * C::TC + j) * 2 + half) * C::THREADS + tid;
  };

  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    // the tile's points [base, base + nvalid) and its network
    int64_t base, nvalid;
    const float *w0 = prm.w0, *bias = prm.bias, *fwd_t = prm.fwd_t, *bwdw = prm.bwd,
                *wout = prm.wout, *bout = prm.bout;
    const float *ffB = prm.ffB, *ff0_t = prm.ff0_t, *ff0 = prm.ff0;
    // the tile's body in a posed grouped launch (its pose is g_T[body]), or -1
    int body = -1;
    if (grouped) {
      int lo = 0, hi = prm.g_nets;               // last k with tile_start[k] <= tile
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prm.g_tile_start[mid] <= tile) lo = mid; else hi = mid;
      }
      const int64_t local = tile - prm.g_tile_start[lo];
      base = prm.g_offsets[lo] + local * C::P;
      nvalid = prm.g_counts[lo] - local * C::P;
      const NetPtrs &np = prm.g_netptrs[lo];
      w0 = np.w0; bias = np.bias; fwd_t = np.fwd_t; bwdw = np.bwd; wout = np.wout; bout = np.bout;
      ffB = np.ffB; ff0_t = np.ff0_t; ff0 = np.ff0;
      if (prm.g_T) body = lo;
    } else {
      base = tile * C::P;
      nvalid = prm.n - base;
    }
    if (nvalid > C::P) nvalid = C::P;

    // ---- the tile's weight panels, in the order they are used, as one stream
    // of KC-row chunks: (ff0_t), fwd_t 1 .. L-1, bwd L-1 .. 1, (ff0) ----
    const int npanels = 2 * (L - 1) + (FF ? 2 : 0);
    int next_panel = 0, next_chunk = 0;          // what stage() copies next
    const float4 *next_src = nullptr;
    auto stage = [&](int slot_index) {
      if (next_panel < npanels) {
        if (next_chunk == 0) {
          int m = next_panel;
          const float *src;
          if (FF && m == 0) {
            src = ff0_t;
          } else {
            if (FF) --m;
            src = m < L - 1 ? fwd_t + (size_t)m * W * W
                            : (m < 2 * (L - 1) ? bwdw + (size_t)(2 * (L - 1) - 1 - m) * W * W : ff0);
          }
          next_src = reinterpret_cast<const float4 *>(src) + tid;
        }
        float4 *dst = reinterpret_cast<float4 *>(Ms + slot_index * C::KC * W) + tid;
        constexpr int kCopies = C::KC * W / 4 / C::THREADS;
        static_assert(C::KC * W / 4 % C::THREADS == 0, "whole copies per thread");
#pragma unroll
        for (int v = 0; v < kCopies; ++v) cp_async16(dst + v * C::THREADS, next_src + v * C::THREADS);
        next_src += C::KC * W / 4;
        if (++next_chunk == C::NCHUNK) {
          next_chunk = 0;
          ++next_panel;
        }
      }
      cp_async_commit();
    };
    static_assert(C::NS == 2, "the ring's slots alternate");
    int q = 0;                                   // slot of the chunk to consume
    stage(0);

    // ---- a1: point load (+ T^{-1}) ----
    if (tid < C::P) {
      int64_t idx = base + tid;
      float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
      if (tid < nvalid) p = prm.pts[idx];
      if (body >= 0 || prm.has_T) {   // p' = T^{-1} p (Sec. 4.2)
        const float *t = body >= 0 ? prm.g_T + (size_t)kBodyFloats * body : prm.Ti;
        float x = t[0] * p.x + t[1] * p.y + t[2] * p.z + t[3];
        float y = t[4] * p.x + t[5] * p.y + t[6] * p.z + t[7];
        float z = t[8] * p.x + t[9] * p.y + t[10] * p.z + t[11];
        p.x = x; p.y = y; p.z = z;
      }
      Ps[tid] = p;
#pragma unroll
      for (int k = 0; k < 4; ++k) dir[tid * 4 + k] = 0.0f;
    }
    __syncthreads();

    // acc[j][h]: column j, point pair h; acc = sum_k X[k][point] M[k][column],
    // the next panel of the stream as M.  All threads call it together.
    float2 acc[C::TC][4];
    auto product = [&]() {
#pragma unroll
      for (int j = 0; j < C::TC; ++j)
#pragma unroll
        for (int h = 0; h < 4; ++h) acc[j][h] = make_float2(0.f, 0.f);
      const float *xk = X + pb;
#pragma unroll 1
      for (int kc = 0; kc < C::NCHUNK; ++kc, q ^= 1) {
        cp_async_wait<0>();
        __syncthreads();          // this chunk is there; the one before and (kc = 0) X are done with
        stage(q ^ 1);
        const float *mk = Ms + q * C::KC * W + cb;
        constexpr int kUnroll = W <= 64 ? 2 : 4;   // (four spill at the narrow widths' 80 registers)
#pragma unroll kUnroll
        for (int k = 0; k < C::KC; ++k, xk += C::XS, mk += W) {
          const float4 xa = *reinterpret_cast<const float4 *>(xk);
          const float4 xb = *reinterpret_cast<const float4 *>(xk + 16);
          float4 wv[C::TC / 4];
          wv[0] = *reinterpret_cast<const float4 *>(mk);
          if (C::TC == 8) wv[C::TC / 4 - 1] = *reinterpret_cast<const float4 *>(mk + 32);
#pragma unroll
          for (int j = 0; j < C::TC; ++j) {
            const float2 w = f2_splat(el4(wv[j / 4], j % 4));
            acc[j][0] = f2_fma(make_float2(xa.x, xa.y), w, acc[j][0]);
            acc[j][1] = f2_fma(make_float2(xa.z, xa.w), w, acc[j][1]);
            acc[j][2] = f2_fma(make_float2(xb.x, xb.y), w, acc[j][2]);
            acc[j][3] = f2_fma(make_float2(xb.z, xb.w), w, acc[j][3]);
          }
        }
      }
      __syncthreads();            // every warp has read X: it may be replaced
    };
    auto store_x = [&](int c, const float (&v)[8]) {
      float *o = X + c * C::XS + pb;
      *reinterpret_cast<float4 *>(o) = make_float4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<float4 *>(o + 16) = make_float4(v[4], v[5], v[6], v[7]);
    };

    const int m = FF ? prm.ff : 0;
    if (FF) {
      // ---- Fourier features gamma(p) (2m = W values) as L0's input tile ----
      // (not unrolled: this phase must not raise the kernel's registers)
#pragma unroll 1
      for (int j = 0; j < C::TC; ++j) {
        const int c = column(j);
        const int fi = c < m ? c : c - m;
        const float bx = ffB[fi * 3 + 0], by = ffB[fi * 3 + 1], bz = ffB[fi * 3 + 2];
#pragma unroll 1
        for (int i = 0; i < C::TP; ++i) {
          const int pr = point(i);
          const float4 p = Ps[pr];
          float sn, cs;
          ff_sincos(bx, by, bz, p.x, p.y, p.z, sn, cs);
          X[c * C::XS + pr] = c < m ? sn : cs;
        }
      }
      product();
    } else {
      // ---- a2: L0 (K = 3) on CUDA cores ----
#pragma unroll
      for (int j = 0; j < C::TC; ++j) {
        const int c = column(j);
        const float w0x = w0[c * 3 + 0], w0y = w0[c * 3 + 1], w0z = w0[c * 3 + 2];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const float4 p = Ps[point(2 * h)], r = Ps[point(2 * h + 1)];
          acc[j][h] = make_float2(fmaf(w0x, p.x, fmaf(w0y, p.y, w0z * p.z)),
                                  fmaf(w0x, r.x, fmaf(w0y, r.y, w0z * r.z)));
        }
      }
    }

    // ---- a3/a4/a5: hidden layers, activation epilogue, output unit ----
    // (the last layer, like the last reverse product below, stands outside its
    // loop, so that the sums over columns take no registers inside it)
    auto activate = [&](int j, float bc, float (&h)[8], float (&s)[8]) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float z = (i & 1 ? acc[j][i / 2].y : acc[j][i / 2].x) + bc;
        act_and_slope(z, beta, inv_beta, prm.relu, h[i], s[i]);
      }
    };
#pragma unroll 1
    for (int l = 0; l < L - 1; ++l) {
      if (l > 0) product();
      const float *b = bias + (size_t)l * W;
      const bool feeds_skip = (skip > 0 && l == skip - 1);
#pragma unroll
      for (int j = 0; j < C::TC; ++j) {
        const int c = column(j);
        float h[8], s[8];
        activate(j, b[c], h, s);
        *slot(l, j, 0) = make_float4(s[0], s[1], s[2], s[3]);
        *slot(l, j, 1) = make_float4(s[4], s[5], s[6], s[7]);
        if (feeds_skip) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float v = h[i];
            if (c >= nshort) {
              const float4 p = Ps[point(i)];
              const int k = c - nshort;
              v = k == 0 ? p.x : k == 1 ? p.y : p.z;
            }
            h[i] = v * kInvSqrt2;
          }
        }
        store_x(c, h);
      }
    }
    if (L > 1) product();
    float fpart[C::TP];
#pragma unroll
    for (int i = 0; i < C::TP; ++i) fpart[i] = 0.0f;
#pragma unroll
    for (int j = 0; j < C::TC; ++j) {
      const int c = column(j);
      const float wo = wout[c];
      float h[8], s[8];
      activate(j, bias[(size_t)(L - 1) * W + c], h, s);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        fpart[i] = fmaf(wo, h[i], fpart[i]);
        h[i] = s[i] * wo;                    // delta_{L-1} = sigmoid' * w_out
      }
      store_x(c, h);
    }

    // f: reduce the partial dot products over the warp's columns
#pragma unroll
    for (int i = 0; i < C::TP; ++i) {
      float v = fpart[i];
#pragma unroll
      for (int o = 1; o < 32; o <<= 2) v += __shfl_xor_sync(0xffffffffu, v, o);   // the bits of lc
      if (lc == 0) red[(cw * C::P + point(i)) * 4 + 3] = v;
    }

    // ---- a6: Jacobian-transpose chain ----
    // d = delta_{l-1} of column j, from the product W_l^T delta_l in acc
    auto reverse_delta = [&](int l, int j, float (&d)[8]) {
      const int c = column(j);
      const float4 s0 = *slot(l - 1, j, 0), s1 = *slot(l - 1, j, 1);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float u = i & 1 ? acc[j][i / 2].y : acc[j][i / 2].x;
        if (skip > 0 && l == skip) {
          u *= kInvSqrt2;
          if (c >= nshort) {                 // direct path to the input
            dir[point(i) * 4 + (c - nshort)] += u;
            u = 0.0f;
          }
        }
        d[i] = el4(i < 4 ? s0 : s1, i & 3) * u;
      }
    };
#pragma unroll 1
    for (int l = L - 1; l >= (FF ? 1 : 2); --l) {
      product();
#pragma unroll
      for (int j = 0; j < C::TC; ++j) {
        float d[8];
        reverse_delta(l, j, d);
        store_x(column(j), d);
      }
    }
    if (FF || L > 1) product();              // W_1^T delta_1, or g_gamma = W_0^T delta_0
    float gp[C::TP][3];
#pragma unroll
    for (int i = 0; i < C::TP; ++i) gp[i][0] = gp[i][1] = gp[i][2] = 0.0f;
    if (!FF) {
      // grad f += delta_0 W_0 (L = 1: delta_0 = sigmoid'(z_0) * w_out sits in X)
#pragma unroll
      for (int j = 0; j < C::TC; ++j) {
        const int c = column(j);
        float d[8];
        if (L > 1) {
          reverse_delta(1, j, d);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) d[i] = X[c * C::XS + point(i)];
        }
        const float wx = w0[c * 3 + 0], wy = w0[c * 3 + 1], wz = w0[c * 3 + 2];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          gp[i][0] = fmaf(d[i], wx, gp[i][0]);
          gp[i][1] = fmaf(d[i], wy, gp[i][1]);
          gp[i][2] = fmaf(d[i], wz, gp[i][2]);
        }
      }
    }
    if (FF) {
      // ---- g_gamma through the feature Jacobian ----
      //   d sin(2 pi b.p)/dp = 2 pi cos(2 pi b.p) b,
      //   d cos(2 pi b.p)/dp = -2 pi sin(2 pi b.p) b
      // park g_gamma in X (each thread its own elements, so no barrier), so
      // that acc is dead while the sines and cosines are evaluated
#pragma unroll
      for (int j = 0; j < C::TC; ++j) {
        const float g[8] = {acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y,
                            acc[j][2].x, acc[j][2].y, acc[j][3].x, acc[j][3].y};
        store_x(column(j), g);
      }
      constexpr float kTwoPi = 6.28318530717958648f;
#pragma unroll 1
      for (int j = 0; j < C::TC; ++j) {
        const int c = column(j);
        const int fi = c < m ? c : c - m;
        const float bx = ffB[fi * 3 + 0], by = ffB[fi * 3 + 1], bz = ffB[fi * 3 + 2];
#pragma unroll
        for (int i = 0; i < C::TP; ++i) {
          const int pr = point(i);
          const float4 p = Ps[pr];
          const float gg = X[c * C::XS + pr];
          float sn, cs;
          ff_sincos(bx, by, bz, p.x, p.y, p.z, sn, cs);
          const float coef = kTwoPi * (c < m ? gg * cs : -gg * sn);
          gp[i][0] = fmaf(coef, bx, gp[i][0]);
          gp[i][1] = fmaf(coef, by, gp[i][1]);
          gp[i][2] = fmaf(coef, bz, gp[i][2]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < C::TP; ++i) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        float v = gp[i][k];
#pragma unroll
        for (int o = 1; o < 32; o <<= 2) v += __shfl_xor_sync(0xffffffffu, v, o);   // the bits of lc
        if (lc == 0) red[(cw * C::P + point(i)) * 4 + k] = v;
      }
    }
    __syncthreads();

    // ---- a7/a8/a9: normalise, collision test, projection ----
    if (tid < C::P) {
      const int64_t idx = base + tid;
      float gx = dir[tid * 4 + 0], gy = dir[tid * 4 + 1], gz = dir[tid * 4 + 2];
      float f = bout[0];
#pragma unroll
      for (int w = 0; w < C::CW; ++w) {
        const float *r = red + (w * C::P + tid) * 4;
        gx += r[0]; gy += r[1]; gz += r[2]; f += r[3];
      }
      if (tid < nvalid) {
        const float nrm = sqrtf(gx * gx + gy * gy + gz * gz);
        float nx = 0.f, ny = 0.f, nz = 0.f;
        if (nrm >= 1e-20f) { nx = gx / nrm; ny = gy / nrm; nz = gz / nrm; }
        if (prm.grad_scale) {
          const float a = prm.grad_scale[idx];
          prm.out_grad[idx] = make_float4(a * gx, a * gy, a * gz, 0.f);
        } else if (!prm.collide) {
          if (prm.raw_gradient) { nx = gx; ny = gy; nz = gz; }
          prm.out_n_sdf[idx] = make_float4(nx, ny, nz, f);
        } else {
          if (body >= 0 || prm.has_T) {   // N rotated by T[:3,:3]
            const float *R = body >= 0 ? prm.g_T + (size_t)kBodyFloats * body + 12 : prm.R;
            float wx = R[0] * nx + R[1] * ny + R[2] * nz;
            float wy = R[3] * nx + R[4] * ny + R[5] * nz;
            float wz = R[6] * nx + R[7] * ny + R[8] * nz;
            nx = wx; ny = wy; nz = wz;
          }
          const bool hit = f < prm.eps;
          float4 p = prm.pts[idx];
          if (hit) {
            const float d = prm.eps - f;
            p.x = fmaf(d, nx, p.x); p.y = fmaf(d, ny, p.y); p.z = fmaf(d, nz, p.z);
          }
          if (prm.out_pts) prm.out_pts[idx] = p;
          if (prm.out_n_sdf) prm.out_n_sdf[idx] = make_float4(nx, ny, nz, f);
          if (prm.out_hit) prm.out_hit[idx] = hit ? 1 : 0;
        }
      }
    }
    __syncthreads();
  }
}

// Host helpers of one (W, PT, FF) instantiation.
template <int W, int PT_, bool FF>
int per_sm_t() {
  using C = Cfg<W, PT_>;
  int per_sm = 1;
  // the occupancy of a kernel above 48 KB of dynamic shared memory is only
  // known once its opt-in attribute is set
  cudaFuncSetAttribute(query_fp32_kernel<W, PT_, FF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)C::SMEM_BYTES);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, query_fp32_kernel<W, PT_, FF>, C::THREADS,
                                                C::SMEM_BYTES);
  return per_sm < 1 ? 1 : per_sm;
}

template <int W, int PT_, bool FF>
cudaError_t launch_t(const QueryParams &p, int grid, cudaStream_t s) {
  using C = Cfg<W, PT_>;
  cudaError_t e = cudaFuncSetAttribute(query_fp32_kernel<W, PT_, FF>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)C::SMEM_BYTES);
  if (e != cudaSuccess) return e;
  query_fp32_kernel<W, PT_, FF><<<grid, C::THREADS, C::SMEM_BYTES, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

#define NSDF_FP32_WIDTHS(X) X(32) X(64) X(128) X(256) X(512)

}  // namespace nsdf
