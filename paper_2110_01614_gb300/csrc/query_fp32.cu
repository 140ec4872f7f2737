// Launchers of the FP32 fused query kernel.  The kernel is in
// query_fp32_kernel.cuh; this file instantiates it for networks without
// Fourier features, query_fp32_ff.cu for networks with them (Sec. 4.3).

#include "query_fp32_kernel.cuh"

namespace nsdf {

// query_fp32_ff.cu
int fp32_ff_per_sm(int width, int pt);
cudaError_t fp32_ff_launch(const QueryParams &p, int pt, int grid, cudaStream_t s);

bool query_fp32_supported(int width) {
  return width == 32 || width == 64 || width == 128 || width == 256 || width == 512;
}

int fp32_tile_points(int width, int pt) {
#define CASE(W) \
  if (width == W) return pt == 4 ? Cfg<W, 4>::P : Cfg<W, 8>::P;
  NSDF_FP32_WIDTHS(CASE)
#undef CASE
  return 0;
}

int fp32_ctas_per_sm(int width, int pt, bool ff) {
  if (ff) return fp32_ff_per_sm(width, pt);
#define CASE(W) \
  if (width == W) return pt == 4 ? per_sm_t<W, 4, false>() : per_sm_t<W, 8, false>();
  NSDF_FP32_WIDTHS(CASE)
#undef CASE
  return 1;
}

// Tile shape of a single-network launch: the small tiles when all of them fit
// on the GPU at once in place of the large ones (more SMs at work), else the large.
Fp32Launch fp32_single_launch(int width, int64_t n, int num_sms, bool ff) {
  if (!query_fp32_supported(width)) return {8, 0};
  const int64_t cap = (int64_t)num_sms * fp32_ctas_per_sm(width, 8, ff);
  const int P4 = fp32_tile_points(width, 4), P8 = fp32_tile_points(width, 8);
  const int64_t tiles4 = (n + P4 - 1) / P4, tiles8 = (n + P8 - 1) / P8;
  if (tiles4 <= cap) return {4, (int)(tiles4 < 1 ? 1 : tiles4)};
  return {8, (int)(tiles8 < cap ? tiles8 : cap)};
}

// The rule where no shape has been set: the small tiles for bodies of at most four
// large tiles on average, whose last tiles would be mostly padding, and for scenes
// whose small tiles all fit on the GPU at once; else the large ones.  Measured, large
// -> small: 1,000 bodies of 40 points at width 64 113 -> 70 us, of 300 points 292 ->
// 267, of 1,000 points 805 -> 807; 8 bodies of 3,000 35 -> 29, of 20,000 146 -> 152;
// 40 bodies of 20 points at width 512 535 -> 300, 100 bodies of 50 points at width
// 256 161 -> 166.
static int grouped_shape(int width, int64_t max_total, int n_nets, int num_sms, bool ff) {
  const int64_t P4 = fp32_tile_points(width, 4), P8 = fp32_tile_points(width, 8);
  if ((max_total + P4 - 1) / P4 + n_nets <= (int64_t)num_sms * fp32_ctas_per_sm(width, 8, ff)) return 4;
  return max_total <= 4 * P8 * n_nets ? 4 : 8;
}

Fp32Launch fp32_grouped_launch(int width, int pt, int cps, int64_t max_total, int n_nets, int num_sms,
                               bool ff) {
  if (pt == 0) pt = grouped_shape(width, max_total, n_nets, num_sms, ff);
  const int P = fp32_tile_points(width, pt);
  const int fit = fp32_ctas_per_sm(width, pt, ff);
  if (cps <= 0 || cps > fit) cps = fit;
  const int64_t max_tiles = (max_total + P - 1) / P + n_nets;
  const int64_t cap = (int64_t)num_sms * cps;
  return {pt, (int)(max_tiles < cap ? max_tiles : cap)};
}

// Where the large tile's slabs are so few that more than an eighth of the SMs would
// have none, the small tile's, twice as many, are faster: 131,077 points in 32 MiB at
// width 512, 8 layers, 68.3 -> 37.4 ms (36 -> 73 CTAs), at width 256, 8 layers, 9.56 ->
// 5.82 ms (73 -> 146); with 146 of 152 SMs at work (width 128, 8 layers) the large tile
// stays, 1.39 ms.
Fp32Launch fp32_bounded_launch(int width, int n_hidden, int64_t n, int num_sms, bool ff, size_t bytes) {
  const Fp32Launch free = fp32_single_launch(width, n, num_sms, ff);
  if (free.grid == 0) return free;
  auto fitting = [&](int pt) -> Fp32Launch {
    const int P = fp32_tile_points(width, pt);
    const int64_t tiles = (n + P - 1) / P, slabs = (int64_t)(bytes / fp32_launch_bytes(width, n_hidden, {pt, 1}));
    int64_t grid = (int64_t)num_sms * fp32_ctas_per_sm(width, pt, ff);
    if (slabs < grid) grid = slabs;
    return {pt, (int)(tiles < grid ? tiles : grid)};
  };
  const Fp32Launch small = fitting(4), large = fitting(8);
  if (free.pt == 4 && small.grid >= free.grid) return free;
  return 8 * (int64_t)large.grid < 7 * (int64_t)num_sms && small.grid > large.grid ? small : large;
}

size_t fp32_launch_bytes(int width, int n_hidden, const Fp32Launch &l) {
  const int slabs = n_hidden > 1 ? n_hidden - 1 : 1;
  return sizeof(float) * (size_t)l.grid * slabs * fp32_tile_points(width, l.pt) * width;
}

// The bound is taken over both tile shapes and every number of CTAs per SM: `n_nets`
// tiles beside the points', of the large shape, at most what is resident.
size_t fp32_scratch_bytes(int width, int n_hidden, int64_t points, int n_nets, int num_sms, bool ff) {
  const int64_t P4 = fp32_tile_points(width, 4), P8 = fp32_tile_points(width, 8);
  const int64_t per_sm4 = P4 * fp32_ctas_per_sm(width, 4, ff), per_sm8 = P8 * fp32_ctas_per_sm(width, 8, ff);
  const int64_t rows = ((points + P8 - 1) / P8 + n_nets) * P8;
  const int64_t cap = num_sms * (per_sm4 > per_sm8 ? per_sm4 : per_sm8);
  const int slabs = n_hidden > 1 ? n_hidden - 1 : 1;
  return sizeof(float) * (size_t)(rows < cap ? rows : cap) * slabs * width;
}

cudaError_t launch_query_fp32_as(const QueryParams &p, const Fp32Launch &l, cudaStream_t s) {
  const int pt = l.pt, grid = l.grid;
  if (p.ff > 0) return fp32_ff_launch(p, pt, grid, s);
#define CASE(W)                                                                           \
  if (p.width == W)                                                                       \
    return pt == 4 ? launch_t<W, 4, false>(p, grid, s) : launch_t<W, 8, false>(p, grid, s);
  NSDF_FP32_WIDTHS(CASE)
#undef CASE
  return cudaErrorInvalidValue;
}

cudaError_t launch_query_fp32(const QueryParams &p, int num_sms, cudaStream_t s) {
  const Fp32Launch l = fp32_single_launch(p.width, p.n, num_sms, p.ff > 0);
  if (l.grid == 0) return cudaErrorInvalidValue;
  return launch_query_fp32_as(p, l, s);
}

}  // namespace nsdf
