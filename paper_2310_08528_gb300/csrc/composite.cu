// Per-tile front-to-back alpha compositing (Eq. 4 with the Gaussian weight of
// Eq. 1).  One 256-thread CTA per 16x16 screen tile (optionally in a given launch
// order, longest lists first), one pixel per thread; warp
// w owns the 8x4 pixel block (w % 2, w / 2) of the tile.  The tile's depth-
// sorted list is walked in batches of 256: each thread gathers one Gaussian into
// shared memory -- position and log2-scaled conic, opacity and colour -- and the
// 8-bit mask of the warp blocks that the ellipse {alpha >= 1/255} can reach.
// Each warp then compacts the batch to the Gaussians whose mask holds its block
// (ballot + popc, order kept) and walks only those; every pixel evaluates Eq. 1
// exactly for them.  The mask is conservative, so it never changes a decision.
// A warp whose pixels have all saturated skips the batch; a CTA stops as soon as
// all of its pixels have (__syncthreads_count).  Batches alternate between two
// staging buffers, so one barrier per batch suffices.
#include "fs4d_internal.cuh"

namespace fs4d {
namespace {

constexpr int kThreads = kTile * kTile;
constexpr int kBatch = kThreads;
constexpr int kWarps = kThreads / 32;
constexpr float kTMin = 1e-4f;
constexpr int kMinBlocks = 4;  // CTAs per SM the register budget must allow
constexpr int kStep = 4;       // Gaussians per step of the walk

// Staged Gaussians, 16 bytes apart in three arrays so that one byte offset finds them all.
constexpr int kSlots = 2 * kBatch + 1;  // two staging buffers and a Gaussian that adds nothing
struct Staged {
  float4 g0[kSlots];    // x, y, a2, c2
  float4 g1[kSlots];    // b2, opacity, red, green
  float4 blue[kSlots];  // .x
};

// One staged batch of m Gaussians (list positions base .. base + m - 1) for the
// calling thread's pixel: the warp compacts the batch to the Gaussians whose mask
// holds its block (ballot, order kept) and walks them kStep at a time -- all weights
// are evaluated before the (sequential, front-to-back) transmittance updates, and the
// list is filled up to a whole step with the Gaussian that adds nothing.  A saturated
// pixel's threshold goes to infinity, so that one comparison decides whether a term
// blends.  AUX: track each pixel's last contributor.
// Bound by instruction issue, so the form of the loop is what counts.  us for the
// compositing of 100,000 Gaussians at 800x800 (with its call) / 300,000 at 1352x1014 / 2M
// at 1920x1080: 52.2 / 201 / 1332 with two terms per step and an exit per pixel (byte
// indices, five CTAs per SM); 49.9 / 189 / 1276 with updates under predicates and one vote
// per step; 47.5 / 184 / 1250 with four terms per step; 40.4 / 169 / 1203 with byte
// offsets into the staging arrays and the registers of four CTAs per SM (eight terms
// per step: 38.9 / 168 / 1258); 38.2 / 164 / 1186 with the threshold; 37.7 / 158 / 1163
// with the offset and red and green as f32x2.  The exponent's two first products and
// 1 - alpha as f32x2 as well: 37.0 / 159 / 1182.
template <bool AUX>
__device__ __forceinline__ void composite_batch(int m, int base, const Staged& st, int buf, const uint32_t* s_mask,
                                                uint32_t* list, int warp, int lane, float fx, float fy, bool& done,
                                                float& T, float& R, float& G, float& B, int& last) {
  const float inf = __int_as_float(0x7f800000);
  float thr = done ? inf : 1.f / 255.f;
  const uint32_t lane_lt = (1u << lane) - 1u;
  int cnt = 0;
  for (int c0 = 0; c0 < m; c0 += 32) {
    const int j = c0 + lane;
    const bool hit = j < m && ((s_mask[j] >> warp) & 1u);
    const uint32_t bal = __ballot_sync(0xffffffffu, hit);
    if (hit) list[cnt + __popc(bal & lane_lt)] = 16u * (uint32_t)(buf * kBatch + j);
    cnt += __popc(bal);
  }
  if (lane < (-cnt & (kStep - 1))) list[cnt + lane] = 16u * (uint32_t)(kSlots - 1);
  __syncwarp();
  for (int i = 0; i < cnt; i += kStep) {
    const uint4 l = *reinterpret_cast<const uint4*>(list + i);
    const uint32_t off[kStep] = {l.x, l.y, l.z, l.w};
    float4 g1[kStep];
    float al[kStep];
#pragma unroll
    for (int u = 0; u < kStep; ++u) {
      const float4 g0 = staged4(st.g0, off[u]);
      g1[u] = staged4(st.g1, off[u]);
      const float2 d = __fadd2_rn(make_float2(g0.x, g0.y), make_float2(-fx, -fy));
      float gauss;
      al[u] = composite_weight(g0, g1[u].x, g1[u].y, d.x, d.y, gauss);
    }
#pragma unroll
    for (int u = 0; u < kStep; ++u) {
      const float Tn = T * (1.f - al[u]);
      const bool hit = al[u] >= thr, go = Tn >= kTMin;
      if (hit && !go) thr = inf;
      if (hit && go) {
        const float w = al[u] * T;
        const float2 rg = __ffma2_rn(make_float2(g1[u].z, g1[u].w), make_float2(w, w), make_float2(R, G));
        R = rg.x;
        G = rg.y;
        B += staged4(st.blue, off[u]).x * w;
        T = Tn;
        if (AUX) last = base + (int)(off[u] >> 4) - buf * kBatch + 1;
      }
    }
    if (__all_sync(0xffffffffu, thr > 1.f)) break;
  }
  done = thr > 1.f;
  __syncwarp();
}

// Stage Gaussian g of a batch into slot k.
__device__ __forceinline__ void stage_gaussian(int k, int slot, uint32_t g, const float2* __restrict__ xy,
                                               const float4* __restrict__ conic_opacity,
                                               const float* __restrict__ rgb, int tx, int ty, Staged& st,
                                               uint32_t* s_mask) {
  const float2 p = xy[g];
  const float4 co = conic_opacity[g];
  st.g0[slot] = composite_coeffs(p, co);
  st.g1[slot] = make_float4(composite_b2(co), co.w, rgb[3 * g], rgb[3 * g + 1]);
  st.blue[slot].x = rgb[3 * g + 2];
  s_mask[k] = block_mask(p, co, composite_exp_threshold(co.w), tx, ty);
}

__device__ __forceinline__ void write_pixel(bool inside, int px, int py, int width, float R, float G, float B,
                                            float T, int last, float* image, float* t_final, int* n_contrib,
                                            bool aux) {
  if (!inside) return;
  const int pix = py * width + px;
  image[3 * pix] = R;
  image[3 * pix + 1] = G;
  image[3 * pix + 2] = B;
  if (aux) {
    if (t_final) t_final[pix] = T;
    if (n_contrib) n_contrib[pix] = last;
  }
}

// Tile lists as [start, end) ranges into a list of Gaussian indices.
template <bool AUX>
__global__ void __launch_bounds__(kThreads, kMinBlocks) composite_kernel(int width, int height, int tiles_x,
                                                            const uint2* __restrict__ ranges,
                                                            const uint32_t* __restrict__ values,
                                                            const float2* __restrict__ xy,
                                                            const float4* __restrict__ conic_opacity,
                                                            const float* __restrict__ rgb, float* __restrict__ image,
                                                            float* __restrict__ t_final, int* __restrict__ n_contrib,
                                                            TileOrder to, int vstride) {
  // two staging buffers: batch i is staged while batch i - 1 may still be read
  __shared__ Staged st;
  __shared__ uint32_t s_maskb[2][kBatch];
  __shared__ __align__(16) uint32_t s_list[kWarps][kBatch];
  if (threadIdx.x == 0) st.g0[kSlots - 1] = st.g1[kSlots - 1] = st.blue[kSlots - 1] = make_float4(0.f, 0.f, 0.f, 0.f);
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int tile = (int)blockIdx.x;
  bool empty = false;
  if (to.order) {
    tile = (int)to.order[blockIdx.x];
  } else if (to.class_count) {  // each warp finds the CTA's place among the length classes
    const uint32_t c = to.class_count[lane];
    uint32_t incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    const int cls = __ffs(__ballot_sync(0xffffffffu, incl > blockIdx.x)) - 1;
    const uint32_t first = __shfl_sync(0xffffffffu, incl - c, cls);
    tile = (int)to.class_tiles[(size_t)cls * to.n_tiles + (blockIdx.x - first)];
    empty = (long long)*to.listed > to.capacity;
  }
  if (to.out && threadIdx.x == 0) to.out[blockIdx.x] = (uint32_t)tile;
  const int tx = tile % tiles_x, ty = tile / tiles_x;
  const int bx0 = tx * kTile + (warp & 1) * 8, by0 = ty * kTile + (warp >> 1) * 4;
  const int px = bx0 + (lane & 7), py = by0 + (lane >> 3);
  const bool inside = px < width && py < height;
  const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
  const uint2 range = ranges[tile];
  const int n = empty ? 0 : (int)(range.y - range.x);

  bool done = !inside;
  float T = 1.f, R = 0.f, G = 0.f, B = 0.f;
  int last = 0;
  for (int base = 0, it = 0; base < n; base += kBatch, ++it) {
    const int b = it & 1;
    const int k = base + (int)threadIdx.x;
    if (k < n)
      stage_gaussian(threadIdx.x, b * kBatch + (int)threadIdx.x, values[(size_t)vstride * (range.x + k)], xy, conic_opacity, rgb, tx, ty, st, s_maskb[b]);
    // one barrier per batch: this batch is staged, the buffer staged next was
    // last read for batch i - 1, which every thread has finished; and if every
    // pixel has saturated the tile is done
    if (__syncthreads_count(done) == kThreads) break;
    if (__all_sync(0xffffffffu, done)) continue;  // warp-uniform
    composite_batch<AUX>(min(kBatch, n - base), base, st, b, s_maskb[b], s_list[warp],
                         warp, lane, fx, fy, done, T, R, G, B, last);
  }
  write_pixel(inside, px, py, width, R, G, B, T, last, image, t_final, n_contrib, AUX);
}

// Tiles straight from the depth order (direct.cu): the tile's list is the set bits
// of its column's and its row's bits, 131072 depth ranks per step (four 16-byte words
// of each per thread, all in flight together).  Up to kQueue ranks of a step go into
// shared memory in order and are staged and blended as the listed tiles' are; a step
// with more is scanned again for each kQueue of them, which keeps the words out of the
// registers that the blending needs.  The walk ends when every pixel has saturated, so
// the far ranks of a covered tile are never looked at; a tile that never saturates
// looks at all of them, which is why the steps are long: 1.49 ms for 2M Gaussians of
// log-scale -2.5 at 1920x1080, 1.85 ms with steps of 32768 ranks (a background tile
// waits for 61 loads in a row instead of 16); 1.16 ms with tighter block masks and the
// walk of four terms per step.
constexpr int kQueue = 2048;
constexpr int kRounds = 4;   // 16-byte words per thread and step

template <bool AUX>
__global__ void __launch_bounds__(kThreads, 4) composite_direct_kernel(const __grid_constant__ DirectArgs a,
                                                                       float* __restrict__ image,
                                                                       float* __restrict__ t_final,
                                                                       int* __restrict__ n_contrib) {
  __shared__ Staged st;
  __shared__ uint32_t s_maskb[2][kBatch];
  __shared__ __align__(16) uint32_t s_list[kWarps][kBatch];
  __shared__ uint32_t s_queue[kQueue];
  __shared__ uint32_t s_warp[2][2][kWarps];
  if (threadIdx.x == 0) st.g0[kSlots - 1] = st.g1[kSlots - 1] = st.blue[kSlots - 1] = make_float4(0.f, 0.f, 0.f, 0.f);
  pdl_wait();
  pdl_trigger();
  const int tx = (int)blockIdx.x % a.tiles_x, row = a.bands.r0[0] + (int)blockIdx.x / a.tiles_x;
  int band = 0;
  while (band + 1 < a.bands.n && a.bands.r0[band + 1] <= row) ++band;
  const float cy = a.bands.cy[band];
  const int ty = row - a.bands.r0[band];  // rows and pixel rows count from the band's first
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int px = tx * kTile + (warp & 1) * 8 + (lane & 7), py = ty * kTile + (warp >> 1) * 4 + (lane >> 3);
  const int gy = py + kTile * a.bands.r0[band];
  const bool inside = px < a.width && gy < a.height;
  const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
  const uint4* col = reinterpret_cast<const uint4*>(a.cols + (size_t)tx * a.words);
  const uint4* rowb = reinterpret_cast<const uint4*>(a.rows + (size_t)row * a.words);
  const int nvec = a.words >> 2;

  bool done = !inside;
  float T = 1.f, R = 0.f, G = 0.f, B = 0.f;
  int last = 0, listed = 0;  // listed: the tile's Gaussians in the steps before this one
  int it = 0;
  bool all_done = false;
  uint32_t w0 = 0;  // list position within the step that the queue starts at
  for (int v0 = 0, pass = 0; v0 < nvec && !all_done; ++pass) {
    // round i holds 16-byte word v0 + i * kThreads + thread: rank order is round by
    // round, thread by thread.  The counts of two rounds (at most 32768 each) are
    // scanned as one packed word.
    uint4 q[kRounds];
    uint32_t c[kRounds];
#pragma unroll
    for (int i = 0; i < kRounds; ++i) {
      const int v = v0 + i * kThreads + (int)threadIdx.x;
      q[i] = make_uint4(0u, 0u, 0u, 0u);
      if (v < nvec) {
        const uint4 x = col[v], y = rowb[v];
        q[i] = make_uint4(x.x & y.x, x.y & y.y, x.z & y.z, x.w & y.w);
      }
      c[i] = __popc(q[i].x) + __popc(q[i].y) + __popc(q[i].z) + __popc(q[i].w);
    }
    const uint32_t p01 = c[0] | (c[1] << 16), p23 = c[2] | (c[3] << 16);
    uint32_t i01 = p01, i23 = p23;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y01 = __shfl_up_sync(0xffffffffu, i01, d), y23 = __shfl_up_sync(0xffffffffu, i23, d);
      if (lane >= d) {
        i01 += y01;
        i23 += y23;
      }
    }
    uint32_t(*sw)[kWarps] = s_warp[pass & 1];  // two buffers: one barrier before they are read, none after
    if (lane == 31) {
      sw[0][warp] = i01;
      sw[1][warp] = i23;
    }
    __syncthreads();
    uint32_t e01 = i01 - p01, e23 = i23 - p23, t01 = 0, t23 = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t y01 = sw[0][w], y23 = sw[1][w];
      if (w < warp) {
        e01 += y01;
        e23 += y23;
      }
      t01 += y01;
      t23 += y23;
    }
    const uint32_t rt[kRounds] = {t01 & 0xffffu, t01 >> 16, t23 & 0xffffu, t23 >> 16};
    const uint32_t ex[kRounds] = {e01 & 0xffffu, e01 >> 16, e23 & 0xffffu, e23 >> 16};
    const uint32_t total = (rt[0] + rt[1]) + (rt[2] + rt[3]);
    if (w0 < total) {
      // this thread's ranks whose list position falls into [w0, w0 + kQueue)
      uint32_t before = 0;
#pragma unroll
      for (int i = 0; i < kRounds; ++i) {
        uint32_t pos = before + ex[i];
        if (pos < w0 + kQueue && pos + c[i] > w0) {
          const uint32_t wd[4] = {q[i].x, q[i].y, q[i].z, q[i].w};
          const uint32_t r0 = 128u * (uint32_t)(v0 + i * kThreads + (int)threadIdx.x);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t m = wd[j];
            while (m) {
              if (pos >= w0 && pos < w0 + kQueue) s_queue[pos - w0] = r0 + 32u * j + (uint32_t)(__ffs(m) - 1);
              ++pos;
              m &= m - 1u;
            }
          }
        }
        before += rt[i];
      }
      __syncthreads();
      const int m = (int)min((uint32_t)kQueue, total - w0);
      for (int b0 = 0; b0 < m; b0 += kBatch, ++it) {
        const int b = it & 1, k = b0 + (int)threadIdx.x;
        if (k < m) {
          const uint32_t rank = s_queue[k];
          const float4 pos = a.s_pos[rank], co = a.s_co[rank];
          const float2 rg = a.s_rg[rank], p = make_float2(pos.x, fmaf(pos.y, pos.z, cy));
          st.g0[b * kBatch + threadIdx.x] = composite_coeffs(p, co);
          st.g1[b * kBatch + threadIdx.x] = make_float4(composite_b2(co), co.w, rg.x, rg.y);
          st.blue[b * kBatch + threadIdx.x].x = pos.w;
          s_maskb[b][threadIdx.x] = block_mask(p, co, composite_exp_threshold(co.w), tx, ty);
        }
        // (as in composite_kernel; the queue is refilled only after the last batch's barrier)
        if (__syncthreads_count(done) == kThreads) {
          all_done = true;
          break;
        }
        if (__all_sync(0xffffffffu, done)) continue;  // warp-uniform
        composite_batch<AUX>(min(kBatch, m - b0), listed + (int)w0 + b0, st, b, s_maskb[b],
                             s_list[warp], warp, lane, fx, fy, done, T, R, G, B, last);
      }
    }
    w0 += kQueue;
    if (w0 >= total) {  // the step's list is done
      listed += (int)total;
      w0 = 0;
      v0 += kRounds * kThreads;
    }
  }
  write_pixel(inside, px, gy, a.width, R, G, B, T, last, image, t_final, n_contrib, AUX);
}

}  // namespace

cudaError_t launch_composite_direct(const DirectArgs& a, float* image, float* t_final, int* n_contrib,
                                    cudaStream_t s) {
  const int rows = a.bands.r0[a.bands.n] - a.bands.r0[0];
  if (a.tiles_x * rows <= 0) return cudaSuccess;
  if (t_final || n_contrib)
    return launch_pdl(composite_direct_kernel<true>, a.tiles_x * rows, kThreads, 0, s, a, image, t_final, n_contrib);
  return launch_pdl(composite_direct_kernel<false>, a.tiles_x * rows, kThreads, 0, s, a, image, t_final, n_contrib);
}

cudaError_t launch_composite(int width, int height, const uint2* ranges, const uint32_t* values, const float2* xy,
                             const float4* conic_opacity, const float* rgb, float* image, float* t_final,
                             int* n_contrib, cudaStream_t s, const TileOrder& order, int values_stride) {
  const int tiles_x = (width + kTile - 1) / kTile, tiles_y = (height + kTile - 1) / kTile;
  if (tiles_x * tiles_y == 0) return cudaSuccess;
  if (t_final || n_contrib)
    return launch_pdl(composite_kernel<true>, tiles_x * tiles_y, kThreads, 0, s, width, height, tiles_x, ranges, values,
                      xy, conic_opacity, rgb, image, t_final, n_contrib, order, values_stride);
  return launch_pdl(composite_kernel<false>, tiles_x * tiles_y, kThreads, 0, s, width, height, tiles_x, ranges, values,
                    xy, conic_opacity, rgb, image, t_final, n_contrib, order, values_stride);
}

}  // namespace fs4d
