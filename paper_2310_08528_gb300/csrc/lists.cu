// Tile lists without a pair sort.  A tile rectangle is a column interval times a row
// interval, so with one bit per depth rank the Gaussians of tile (tx, ty), in depth
// order, are the set bits of columns[tx] & rows[ty]: exactly the order a stable sort of
// (tile | depth) keys gives.  Three kernels:
//   gather  one thread per Gaussian: its depth rank (from the sorted order, or within its
//           depth bucket), the rectangle and what the compositing reads copied into rank
//           order; pair count and slots;
//   bits    the bit rows, by ballots over 32 ranks or one bit at a time;
//   list    one CTA per tile, each warp an eighth of the ranks, 4096 ranks per step (a
//           16-byte word of each bit row per lane): counted, placed and written.
// The lists lie anywhere (an atomic allocation per tile), each tile under its length class
// for the compositing to take the longest first.  Lists with keys in tile order
// (fs4d_bin_sort) are copied from there once the tile counts have been scanned.
//
// Culled lists: the rectangle is cut to the bounding box of the ellipse {alpha >= 1/255},
// once per Gaussian.  (The exact test of every tile against the ellipse, per pair, took
// more than the shorter lists save: 150 us of a 300k room's frame.)
//
// The binning stage against one bit per (tile, rank) with an atomic OR per pair, a tile
// scan and an extraction pass: 300k room at 1352x1014 103 against 170 us, 100k object at
// 800x800 29.7 against 33.8 (gather 6.7, bits 6.4, list 12.4), 2000 Gaussians 13.3 against 17.4.
#include "fs4d_internal.cuh"

namespace fs4d {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kRowsPerCta = 256;    // bit rows per CTA of the bits kernel

// The rectangle of a projected Gaussian cut to the tiles that have a pixel centre within
// the bounding box of its ellipse {alpha >= 1/255}: d^T K d <= S, a 0.4% + 2e-3 margin
// over the compositing's own bound, reaches sqrt(S C / det) in x and sqrt(S A / det) in y
// (1e-3 of it and 0.01 pixels for the rounding).  Without a usable bound the rectangle
// stays.
__device__ __forceinline__ int4 cut_rect(int4 r, float2 p, float4 co) {
  const float thr = composite_exp_threshold(co.w);
  if (!(thr < 0.f)) return make_int4(0, 0, 0, 0);  // alpha never reaches 1/255
  const float det = conic_det(co);
  if (!conic_bounded(co, det)) return r;
  const float S = (-2.f * thr * 1.004f + 2e-3f) / det;
  const float hx = sqrtf(S * co.z) * 1.001f + 0.01f, hy = sqrtf(S * co.x) * 1.001f + 0.01f;
  if (!(hx < 1e6f && hy < 1e6f)) return r;
  // tile t has pixel centres 16 t + 0.5 .. 16 t + 15.5
  const int x0 = (int)ceilf((p.x - hx - 15.5f) * (1.f / kTile)), x1 = (int)floorf((p.x + hx - 0.5f) * (1.f / kTile)) + 1;
  const int y0 = (int)ceilf((p.y - hy - 15.5f) * (1.f / kTile)), y1 = (int)floorf((p.y + hy - 0.5f) * (1.f / kTile)) + 1;
  r = make_int4(max(r.x, x0), max(r.y, y0), min(r.z, x1), min(r.w, y1));
  return r.z > r.x && r.w > r.y ? r : make_int4(0, 0, 0, 0);
}

// Bound by the gathers' latency: everything is requested at once after the index.  The
// words of a CTA are in shared memory while their ranks are counted (an object of 20,000
// Gaussians has about 50 per bucket).
__global__ void __launch_bounds__(kThreads) gather_kernel(const __grid_constant__ ListArgs a) {
  __shared__ uint32_t s_warp[kWarps], s_sum[kWarps], s_slot;
  __shared__ unsigned long long s_kv[kThreads + 2 * kBucketMost];
  pdl_wait();
  pdl_trigger();
  const int i = blockIdx.x * kThreads + (int)threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int pos = i;  // depth rank
  uint32_t g = 0, cnt = 0;
  bool live = i < a.n;
  if (a.buckets.start && a.buckets.start[kBuckets + 1]) {
    // grouped by depth bucket: the rank of a word is its bucket's start plus the smaller
    // words (depth, then index) of the bucket; the CTA's words lie in whole buckets
    const uint32_t seen = a.buckets.start[kBuckets], i0 = blockIdx.x * kThreads;
    const unsigned long long* kv = a.buckets.bucketed;
    live = (uint32_t)i < seen;
    uint32_t lo = 0;
    if (i0 < seen) {
      lo = a.buckets.start[depth_bucket((uint32_t)(kv[i0] >> 32))];
      const uint32_t hi = a.buckets.start[depth_bucket((uint32_t)(kv[min(i0 + kThreads, seen) - 1] >> 32)) + 1];
      for (uint32_t j = lo + threadIdx.x; j < hi; j += kThreads) s_kv[j - lo] = kv[j];
    }
    __syncthreads();
    if (live) {
      const unsigned long long w = s_kv[(uint32_t)i - lo];
      const int b = depth_bucket((uint32_t)(w >> 32));
      const uint32_t s0 = a.buckets.start[b], s1 = a.buckets.start[b + 1];
      uint32_t less = 0;
#pragma unroll 8
      for (uint32_t j = s0 - lo; j < s1 - lo; ++j) less += s_kv[j] < w ? 1u : 0u;
      pos = (int)(s0 + less);
      g = (uint32_t)w;
    } else if (i < a.n) {
      a.s_rect[i] = make_int4(0, 0, 0, 0);  // no Gaussian of this rank
    }
  } else if (live) {
    const uint32_t* order = (a.order_sel && *a.order_sel) ? a.order_alt : a.order;
    g = min(order[i], (uint32_t)a.n - 1u);  // (a sort whose wait gave up leaves anything there)
  }
  int4 cut = make_int4(0, 0, 0, 0);
  if (live) {
    if (a.order_out) a.order_out[pos] = g;
    const int4 r = a.rect[g];
    cnt = (uint32_t)max(0, r.z - r.x) * (uint32_t)max(0, r.w - r.y);
    cut = cnt ? r : cut;
    if (a.s_xy) {
      const float2 p = a.xy[g];
      const float4 co = a.conic_opacity[g];
      const float red = a.rgb[3 * (size_t)g], gr = a.rgb[3 * (size_t)g + 1], bl = a.rgb[3 * (size_t)g + 2];
      a.s_xy[pos] = p;
      a.s_co[pos] = co;
      a.s_rgb[3 * (size_t)pos] = red;
      a.s_rgb[3 * (size_t)pos + 1] = gr;
      a.s_rgb[3 * (size_t)pos + 2] = bl;
      if (a.cull && cnt) cut = cut_rect(r, p, co);
    }
    a.s_rect[pos] = cut;
  }
  // the pairs of the rectangles; a saved frame's slots, one per tile of the cut rectangle
  // (each Gaussian's consecutive, anywhere: an atomic per CTA)
  const uint32_t sum = __reduce_add_sync(0xffffffffu, cnt);
  const uint32_t slots = a.offsets ? (uint32_t)(cut.z - cut.x) * (uint32_t)(cut.w - cut.y) : 0u;
  uint32_t incl = slots;
  if (a.offsets) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
  }
  if (lane == 31) {
    s_sum[warp] = sum;
    s_warp[warp] = incl;
  }
  __syncthreads();
  uint32_t before = 0, total = 0, pairs = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t y = s_warp[w];
    if (w < warp) before += y;
    total += y;
    pairs += s_sum[w];
  }
  if (threadIdx.x == 0) {
    if (pairs) atomicAdd(&a.num_pairs[0], pairs);
    s_slot = total ? atomicAdd(&a.num_pairs[2], total) : 0u;
  }
  if (!a.offsets) return;
  __syncthreads();
  if (live) {
    const uint32_t first = s_slot + before + incl - slots;
    a.offsets[g] = first;
    a.rect[g] = cut;
    a.s_slot[pos] = make_int4(cut.x, cut.y, cut.z - cut.x, (int)first);
  }
}

// 256 ranks (one word of each of eight warps: a whole 32-byte sector of each bit row) and
// 256 bit rows per CTA, collected in shared memory.  A warp of small rectangles sets its
// bits one at a time; one whose rectangles span an eighth of the bit rows or more takes a
// ballot per bit row instead (a 300k room: 34 us with ballots alone).
__global__ void __launch_bounds__(kThreads) bits_kernel(const __grid_constant__ ListArgs a) {
  __shared__ uint32_t s_bits[kRowsPerCta][kWarps];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pos = blockIdx.x * kThreads + (int)threadIdx.x;
  int4 r = make_int4(0, 0, 0, 0);
  if (pos < a.n) r = a.s_rect[pos];
  if (r.z <= r.x || r.w <= r.y) r = make_int4(0, 0, 0, 0);
  const uint32_t rows = (uint32_t)a.tiles_x + (uint32_t)a.tiles_y;  // bit rows: the columns of tiles, then the rows
  const uint32_t span = __reduce_max_sync(0xffffffffu, (uint32_t)(r.z - r.x)) +
                        __reduce_max_sync(0xffffffffu, (uint32_t)(r.w - r.y));
  const bool ballots = span > rows / 8;
  for (uint32_t c0 = blockIdx.y * (uint32_t)kRowsPerCta; c0 < rows; c0 += gridDim.y * (uint32_t)kRowsPerCta) {
    const int m = (int)min((uint32_t)kRowsPerCta, rows - c0);
    // this lane's intervals of the CTA's bit rows
    auto local = [&](long long v) { return (int)min(max(v - (long long)c0, 0ll), (long long)m); };
    const int x0 = local(min(max(r.x, 0), a.tiles_x)), x1 = local(min(max(r.z, 0), a.tiles_x));
    const int y0 = local((long long)a.tiles_x + max(r.y, 0)), y1 = local((long long)a.tiles_x + max(r.w, 0));
    __syncthreads();  // the previous rows have been written out
    if (ballots) {
      for (int q = 0; q < m; ++q) {
        const uint32_t bal = __ballot_sync(0xffffffffu, (q >= x0 && q < x1) || (q >= y0 && q < y1));
        if (lane == (q & 31)) s_bits[q][warp] = bal;
      }
    } else {
      for (int q = lane; q < m; q += 32) s_bits[q][warp] = 0;
      __syncwarp();
      for (int q = x0; q < x1; ++q) atomicOr(&s_bits[q][warp], 1u << lane);
      for (int q = y0; q < y1; ++q) atomicOr(&s_bits[q][warp], 1u << lane);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m * kWarps; i += kThreads) {
      const int q = i / kWarps, w = i % kWarps;
      if (blockIdx.x * kWarps + w < a.words)
        a.bits[(size_t)(c0 + q) * a.words + blockIdx.x * kWarps + w] = s_bits[q][w];
    }
  }
}

// One tile per CTA, the ranks in eight consecutive shares, one per warp.  The words of the
// tile (column and row ANDed) are needed twice, to count the list and, once it has its
// place, to write it.  In between they stay in registers (REGS: four 16-byte words per
// lane, up to 131072 Gaussians) or are read again.  100k object: 12.4 us with registers,
// 16.3 read again; 300k room, about 50 instructions per 4096 ranks and a dozen per pair:
// 74 us read again, 77 with the words in shared memory, 117 with twelve words in registers
// (two CTAs per SM).
constexpr int kRegWords = 4;

template <bool REGS>
__global__ void __launch_bounds__(kThreads) list_kernel(const __grid_constant__ ListArgs a) {
  __shared__ uint32_t s_cnt[kWarps], s_start, s_fits;
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tile = blockIdx.x;
  const int ty = (int)(tile / (uint32_t)a.tiles_x), tx = (int)(tile - (uint32_t)ty * (uint32_t)a.tiles_x);
  const int nvec = a.words >> 2, per = (nvec + kWarps - 1) / kWarps;
  const int v0 = min(nvec, per * warp), v1 = min(nvec, v0 + per);
  const uint4* col = reinterpret_cast<const uint4*>(a.bits + (size_t)tx * a.words);
  const uint4* row = reinterpret_cast<const uint4*>(a.bits + ((size_t)a.tiles_x + ty) * a.words);
  auto word = [&](int v) {
    if (v >= v1) return make_uint4(0u, 0u, 0u, 0u);
    const uint4 x = col[v], y = row[v];
    return make_uint4(x.x & y.x, x.y & y.y, x.z & y.z, x.w & y.w);
  };
  auto ones = [](const uint4& q) { return (uint32_t)(__popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w)); };
  uint4 q[kRegWords];
  uint32_t cnt = 0;
  if constexpr (REGS) {
#pragma unroll
    for (int k = 0; k < kRegWords; ++k) {
      q[k] = word(v0 + 32 * k + lane);
      cnt += ones(q[k]);
    }
  } else {
#pragma unroll 4
    for (int v = v0 + lane; v < v1; v += 32) cnt += ones(word(v));
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) s_cnt[warp] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t total = 0;
    for (int w = 0; w < kWarps; ++w) total += s_cnt[w];
    const uint32_t start = total ? atomicAdd(&a.num_pairs[1], total) : 0u;
    const bool fits = (long long)start + total <= a.capacity;
    if (a.class_count) {
      const int cls = total ? __clz((int)total) - 1 : 31;  // 30 - floor(log2 total), empty tiles last
      a.class_tiles[(size_t)cls * a.n_tiles + atomicAdd(&a.class_count[cls], 1u)] = tile;
    }
    a.ranges[tile] = total && fits ? make_uint2(start, start + total) : make_uint2(0u, 0u);
    if (a.tile_count) a.tile_count[tile] = total;
    if (!fits && a.report_overflow) atomicOr(a.status, kStatusCapacity);
    s_start = start;
    s_fits = fits;
  }
  __syncthreads();
  if (!s_fits || cnt == 0) return;
  uint32_t at = s_start;
  for (int w = 0; w < warp; ++w) at += s_cnt[w];
  auto write = [&](const uint4& w, int v) {  // the step's ranks, lane by lane
    const uint32_t c = ones(w);
    if (!__any_sync(0xffffffffu, c != 0)) return;
    uint32_t incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    uint32_t* out = a.values + at + (incl - c);
    const uint32_t r0 = 128u * (uint32_t)v;
    unsigned long long lo = w.x | ((unsigned long long)w.y << 32), hi = w.z | ((unsigned long long)w.w << 32);
    while (lo) {
      *out++ = r0 + (uint32_t)(__ffsll((long long)lo) - 1);
      lo &= lo - 1;
    }
    while (hi) {
      *out++ = r0 + 64u + (uint32_t)(__ffsll((long long)hi) - 1);
      hi &= hi - 1;
    }
    at += __shfl_sync(0xffffffffu, incl, 31);
  };
  if constexpr (REGS) {
#pragma unroll
    for (int k = 0; k < kRegWords; ++k) write(q[k], v0 + 32 * k + lane);
  } else {
    for (int w0 = v0; w0 < v1; w0 += 32) write(word(w0 + lane), w0 + lane);
  }
}

// Lists of depth ranks at their places (ranges) into lists of Gaussians with keys in tile
// order (out).
__global__ void __launch_bounds__(kThreads) list_keys_kernel(const __grid_constant__ ListArgs a,
                                                             const uint2* __restrict__ out,
                                                             uint32_t* __restrict__ values,
                                                             unsigned long long* __restrict__ keys) {
  pdl_wait();
  pdl_trigger();
  const uint32_t tile = blockIdx.x;
  const uint2 from = a.ranges[tile], to = out[tile];
  if (to.y <= to.x) return;  // empty, or the pairs overflow the buffers
  const uint32_t* order = a.order_out;
  const uint32_t cnt = min(to.y - to.x, from.y - from.x), most = (uint32_t)a.n - 1u;
  constexpr int kU = 4;
  for (uint32_t i0 = threadIdx.x; i0 < cnt; i0 += kU * kThreads) {
    uint32_t g[kU], d[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {  // (ranks are < n: the clamp only guards the gathers)
      const uint32_t i = i0 + u * kThreads;
      g[u] = i < cnt ? min(a.values[from.x + i], most) : 0u;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) g[u] = order[g[u]];
#pragma unroll
    for (int u = 0; u < kU; ++u) d[u] = __float_as_uint(a.depth[g[u]]);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const uint32_t i = i0 + u * kThreads;
      if (i < cnt) {
        values[to.x + i] = g[u];
        keys[to.x + i] = ((unsigned long long)tile << 32) | d[u];
      }
    }
  }
}

}  // namespace

int bitmap_words(int n) { return ((n + 127) / 128) * 4; }

cudaError_t launch_tile_bits(const ListArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (a.words < bitmap_words(a.n) || (a.words & 3)) return cudaErrorInvalidValue;
  cudaError_t e = launch_pdl(gather_kernel, (unsigned)((a.n + kThreads - 1) / kThreads), kThreads, 0, s, a);
  if (e != cudaSuccess) return e;
  const long long rows = (long long)a.tiles_x + a.tiles_y, y = (rows + kRowsPerCta - 1) / kRowsPerCta;
  return launch_pdl_2d(bits_kernel, dim3((unsigned)((a.words + kWarps - 1) / kWarps), (unsigned)(y < 65535 ? y : 65535)),
                       kThreads, 0, s, a);
}

cudaError_t launch_tile_lists(const ListArgs& a, cudaStream_t s) {
  const unsigned grid = (unsigned)a.n_tiles;
  return a.words <= 4 * 32 * kWarps * kRegWords ? launch_pdl(list_kernel<true>, grid, kThreads, 0, s, a)
                                                : launch_pdl(list_kernel<false>, grid, kThreads, 0, s, a);
}

cudaError_t launch_tile_keys(const ListArgs& a, const uint2* out, uint32_t* values, unsigned long long* keys,
                             cudaStream_t s) {
  return launch_pdl(list_keys_kernel, (unsigned)a.n_tiles, kThreads, 0, s, a, out, values, keys);
}

}  // namespace fs4d
