// Binning of the frames that are composited straight from the depth order: frames
// whose Gaussians cover so many tiles that listing every (tile, Gaussian) pair costs
// far more than the pixels read (2M Gaussians of log-scale -2.5 at 1920x1080: 1.35e9
// pairs, of which a tile blends the first one or two thousand of its 165,000 before
// its pixels saturate).
//
// A tile rectangle is a column interval times a row interval, so the list of tile
// (tx, ty) in depth order is the set bits of columns[tx] & rows[ty] with one bit per
// depth rank: tiles_x + tiles_y bit rows (47 MB for that frame) in place of 8 bytes
// per pair, no pair sort, and nothing to size by the number of pairs.  At 1920x1080 /
// 2M the binning and pair sort of three bands took 27.6 ms (emission 6.3, sort
// 21.3); the pair counts take 17 us and the bit rows 181.
#include "fs4d_internal.cuh"

namespace fs4d {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kWordsPerWarp = 4;
constexpr int kWordsPerCta = kWarps * kWordsPerWarp;  // 32 words: a 128-byte line of every bit row
constexpr int kRowsPerFlush = 64;

// Tile rows [y0, y1) of a Gaussian within a band, relative to the band's first row:
// the projection's own arithmetic with the band's principal point.
__device__ __forceinline__ void band_rows(float fpy, float iz, float fr, float cy, int n_rows, int& y0, int& y1) {
  const float v = fmaf(fpy, iz, cy);
  y0 = (int)floorf((v - fr) * (1.f / kTile));
  y1 = (int)floorf((v + fr) * (1.f / kTile)) + 1;
  y0 = min(n_rows, max(0, y0));
  y1 = min(n_rows, max(0, y1));
}

// Tile pairs of each band: the sum of the rectangles' areas.  Streams 28 bytes per
// Gaussian once (2M: 56 MB).
__global__ void __launch_bounds__(kThreads) band_pairs_kernel(const __grid_constant__ DirectArgs a,
                                                              unsigned long long* __restrict__ pairs) {
  __shared__ unsigned long long s_sum[kMaxBands];
  for (int b = threadIdx.x; b < kMaxBands; b += kThreads) s_sum[b] = 0;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  for (int g0 = blockIdx.x * kThreads; g0 < a.n; g0 += gridDim.x * kThreads) {
    const int g = g0 + (int)threadIdx.x;
    int w = 0;
    float fr = 0.f;
    float2 yp = make_float2(0.f, 0.f);
    if (g < a.n) {
      const int rad = a.radius[g];
      if (rad > 0) {
        const int4 r = a.rect[g];
        w = r.z - r.x;
        fr = (float)rad;
        yp = a.y_parts[g];
      }
    }
    for (int b = 0; b < a.bands.n; ++b) {
      int y0, y1;
      band_rows(yp.x, yp.y, fr, a.bands.cy[b], a.bands.r0[b + 1] - a.bands.r0[b], y0, y1);
      uint32_t c = w > 0 && y1 > y0 ? (uint32_t)w * (uint32_t)(y1 - y0) : 0u;  // (at most 2^18 tiles a warp lane)
      c = __reduce_add_sync(0xffffffffu, c);
      if ((threadIdx.x & 31) == 0 && c) atomicAdd(&s_sum[b], (unsigned long long)c);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < a.bands.n; b += kThreads)
    if (s_sum[b]) atomicAdd(&pairs[b], s_sum[b]);
}

// The bit rows, 1024 depth ranks per CTA: a warp holds 32 ranks in its lanes and
// takes one ballot per bit row; 64 rows of 32 words are collected in shared memory
// and written as whole 128-byte lines.  Bound by the ballots (about five instructions
// per row and 32 ranks).  FIRST also writes the column rows and copies what the
// compositing reads of each Gaussian into depth-rank order.
template <bool FIRST>
__global__ void __launch_bounds__(kThreads) axis_bits_kernel(const __grid_constant__ DirectArgs a) {
  __shared__ uint32_t s_bits[kRowsPerFlush][kWordsPerCta];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int word0 = blockIdx.x * kWordsPerCta;
  const uint32_t* order = (a.order_sel && *a.order_sel) ? a.order_alt : a.order;
  int x0[kWordsPerWarp], x1[kWordsPerWarp];
  float fr[kWordsPerWarp], fpy[kWordsPerWarp], iz[kWordsPerWarp];
#pragma unroll
  for (int k = 0; k < kWordsPerWarp; ++k) {
    const int pos = 32 * (word0 + kWordsPerWarp * warp + k) + lane;
    x0[k] = x1[k] = 0;
    fr[k] = fpy[k] = iz[k] = 0.f;
    if (pos < a.n) {
      const uint32_t g = min(order[pos], (uint32_t)a.n - 1u);  // (a sort whose wait gave up leaves anything there)
      const int rad = a.radius[g];
      if (rad > 0) {  // (an invisible Gaussian has no bits, so its copies are never read)
        const int4 r = a.rect[g];
        const float2 yp = a.y_parts[g];
        x0[k] = r.x;
        x1[k] = r.z;
        fr[k] = (float)rad;
        fpy[k] = yp.x;
        iz[k] = yp.y;
        if (FIRST) {
          a.s_pos[pos] = make_float4(a.xy[g].x, yp.x, yp.y, a.rgb[3 * g + 2]);
          a.s_co[pos] = a.conic_opacity[g];
          a.s_rg[pos] = make_float2(a.rgb[3 * g], a.rgb[3 * g + 1]);
        }
      }
    }
  }
  // rows [first, first + count) of `out`, bit row r being lo[k] <= r - off < hi[k] in lane's word k
  auto rows_of = [&](uint32_t* out, int first, int count, const int (&lo)[kWordsPerWarp],
                     const int (&hi)[kWordsPerWarp]) {
    for (int f = 0; f < count; f += kRowsPerFlush) {
      const int m = min(kRowsPerFlush, count - f);
      __syncthreads();  // the previous flush has been written out
#pragma unroll
      for (int k = 0; k < kWordsPerWarp; ++k)
        for (int r = 0; r < m; ++r) {
          const uint32_t bal = __ballot_sync(0xffffffffu, f + r >= lo[k] && f + r < hi[k]);
          if (lane == (r & 31)) s_bits[r][kWordsPerWarp * warp + k] = bal;
        }
      __syncthreads();
      for (int r = warp; r < m; r += kWarps)
        if (word0 + lane < a.words) out[(size_t)(first + f + r) * a.words + word0 + lane] = s_bits[r][lane];
    }
  };
  if (FIRST) rows_of(a.cols, 0, a.tiles_x, x0, x1);
  for (int b = 0; b < a.bands.n; ++b) {
    int y0[kWordsPerWarp], y1[kWordsPerWarp];
    const int count = a.bands.r0[b + 1] - a.bands.r0[b];
#pragma unroll
    for (int k = 0; k < kWordsPerWarp; ++k) {
      band_rows(fpy[k], iz[k], fr[k], a.bands.cy[b], count, y0[k], y1[k]);
      if (x1[k] <= x0[k]) y0[k] = y1[k] = 0;
    }
    rows_of(a.rows, a.bands.r0[b], count, y0, y1);
  }
}

}  // namespace

cudaError_t launch_band_pairs(const DirectArgs& a, unsigned long long* pairs, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  const int need = (a.n + kThreads - 1) / kThreads, most = 8 * device_sm_count();
  return launch_pdl(band_pairs_kernel, need < most ? need : most, kThreads, 0, s, a, pairs);
}

cudaError_t launch_axis_bits(const DirectArgs& a, bool first, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (a.words < bitmap_words(a.n)) return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)((a.words + kWordsPerCta - 1) / kWordsPerCta);
  return first ? launch_pdl(axis_bits_kernel<true>, grid, kThreads, 0, s, a)
               : launch_pdl(axis_bits_kernel<false>, grid, kThreads, 0, s, a);
}

}  // namespace fs4d
