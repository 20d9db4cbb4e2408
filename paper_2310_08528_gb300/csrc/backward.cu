// Backward of the render path (training, Sec. 4.3): the chain rule of
// compositing (Eq. 4 with Eq. 1) and EWA projection (Eq. 2, Eq. 3) with SH colour.
// Float32 throughout.
//
//  composite_bwd_kernel  one CTA per tile, one pixel per thread, walking the
//      tile's list back to front from each pixel's last blended term.  The
//      contributions of the 256 pixels to each Gaussian are summed inside the
//      CTA (warp shuffles, then shared-memory adds) and written ONCE per
//      (tile, Gaussian) pair into that pair's slot, so no
//      global atomics are needed: a Gaussian's slots are contiguous (offsets[g] ...
//      offsets[g] + rect area).
//  project_bwd_kernel    one thread per Gaussian: sums its pair slots, then
//      back-propagates through the conic inverse, Sigma' = A A^T + 0.3 I with
//      A = J W R S, the quaternion normalisation, the perspective Jacobian, the
//      projected mean and the SH colour.
// The deformation's backward and the weight gradients are in mlp_bwd.cu.
#include "fs4d_internal.cuh"

namespace fs4d {
namespace {

constexpr int kBatch = kTile * kTile;
constexpr float kAlphaMax = 0.99f;
constexpr float kGuard = 1.3f;

// ------------------------------------------------------------------ compositing

// The warp's sums of the nine per-lane values of two terms with 21 shuffles (45 each one
// by one): values 0..7 of both are halved at each of the offsets 16, 8, 4, 2 (a lane keeps
// one half and sends the other to its partner) and the last one summed over offset 1, so
// an even lane returns the sum of value (lane / 2) % 8 of term a (lanes 0..15) or b; the
// sums of value 8 come back in s8 (a's in the lower half warp, b's in the upper).
__device__ __forceinline__ float warp_sum18(const float (&a)[kPairGrad], const float (&b)[kPairGrad], unsigned lane,
                                            float& s8) {
  static_assert(kPairGrad == 9, "eight halved values and one summed whole");
  float h8[8], h4[4], h2[2];
  const bool u16 = (lane & 16u) != 0u, u8 = (lane & 8u) != 0u, u4 = (lane & 4u) != 0u, u2 = (lane & 2u) != 0u;
#pragma unroll
  for (int i = 0; i < 8; ++i) h8[i] = (u16 ? b[i] : a[i]) + __shfl_xor_sync(0xffffffffu, u16 ? a[i] : b[i], 16);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    h4[i] = (u8 ? h8[i + 4] : h8[i]) + __shfl_xor_sync(0xffffffffu, u8 ? h8[i] : h8[i + 4], 8);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    h2[i] = (u4 ? h4[i + 2] : h4[i]) + __shfl_xor_sync(0xffffffffu, u4 ? h4[i] : h4[i + 2], 4);
  float h1 = (u2 ? h2[1] : h2[0]) + __shfl_xor_sync(0xffffffffu, u2 ? h2[0] : h2[1], 2);
  h1 += __shfl_xor_sync(0xffffffffu, h1, 1);
  float w = (u16 ? b[8] : a[8]) + __shfl_xor_sync(0xffffffffu, u16 ? a[8] : b[8], 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  s8 = w;
  return h1;
}

// The state of a pixel on its way back to front.
struct PixelBack {
  float T;                 // transmittance behind the current term
  float b0, b1, b2;        // the colour blended behind it
  float dC0, dC1, dC2;     // dL/dC
};

// The gradients of one blended term (alpha > 0) at offset (dx, dy), zero otherwise.  The
// products are rounded per pixel, the opacity's factor included, in this order: a training
// step's first Adam updates take the sign of a gradient alone, so another rounding (the
// opacity multiplied into the sums; col T - b divided once) changes the step of the plane
// cells whose sum cancels below it.  Selects, no branch: nine values under a divergent
// branch took 549 us where selects took 535.
__device__ __forceinline__ void term_grads(PixelBack& p, float alpha, float G, const float4& co, const float4& col,
                                           float dx, float dy, float (&gr)[kPairGrad]) {
  const bool on = alpha > 0.f;
  const float inv = 1.f / (1.f - alpha);
  const float Ti = p.T * inv;
  const float c0 = col.x, c1 = col.y, c2 = col.z;
  const float dalpha =
      p.dC0 * (c0 * Ti - p.b0 * inv) + p.dC1 * (c1 * Ti - p.b1 * inv) + p.dC2 * (c2 * Ti - p.b2 * inv);
  const float w = alpha * Ti;
  gr[6] = on ? p.dC0 * w : 0.f;
  gr[7] = on ? p.dC1 * w : 0.f;
  gr[8] = on ? p.dC2 * w : 0.f;
  if (on) {
    p.b0 += c0 * w;
    p.b1 += c1 * w;
    p.b2 += c2 * w;
    p.T = Ti;
  }
  const bool grad = on && co.w * G <= kAlphaMax;
  const float dpow = grad ? dalpha * co.w * G : 0.f;
  gr[0] = -dpow * (co.x * dx + co.y * dy);
  gr[1] = -dpow * (co.z * dy + co.y * dx);
  gr[2] = -0.5f * dpow * dx * dx;
  gr[3] = -dpow * dx * dy;
  gr[4] = -0.5f * dpow * dy * dy;
  gr[5] = grad ? dalpha * G : 0.f;
}

// Bit w set iff some pixel centre of the 16x2 pixel rows (2w, 2w + 1) of tile (tx, ty), warp
// w's pixels, may reach alpha >= 1/255: block_mask's column intervals and margins, per pair
// of rows.
__device__ __forceinline__ uint32_t row_pair_mask(float2 p, float4 co, float thr, int tx, int ty) {
  if (!(thr < 0.f)) return 0u;
  const float A = co.x, B = co.y, C = co.z, det = conic_det(co);
  if (!conic_bounded(co, det)) return 0xffu;
  const float s = -2.f * thr * 1.002f + 1e-3f;
  const float X0 = (float)(tx * kTile) + 0.5f - p.x, Y0 = (float)(ty * kTile) + 0.5f - p.y;
  const float iA = 1.f / A, sd = s / det, k = B * iA, wA = s * iA, wd = det * iA * iA;
  const float hx = sqrt_approx(sd * C), hy = sqrt_approx(sd * A) * 1.00001f + 0.01f;
  const float yr = -B / C * hx;  // the row of the greatest column
  const float slack = 1e-5f * hx + 0.01f;
  uint32_t mask = 0u;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float ya = Y0 + (float)(2 * r), yb = ya + 1.f;
    const float a = fmaxf(ya, -hy), b = fminf(yb, hy);
    const float va = sqrt_approx(fmaxf(0.f, wA - wd * a * a)), vb = sqrt_approx(fmaxf(0.f, wA - wd * b * b));
    float hi = fmaxf(va - k * a, vb - k * b), lo = fminf(-va - k * a, -vb - k * b);
    if (yr >= a && yr <= b) hi = hx;
    if (-yr >= a && -yr <= b) lo = -hx;
    if (!(a > b) && !(hi + slack < X0) && !(lo - slack > X0 + 15.f)) mask |= 1u << r;
  }
  return mask;
}

// One CTA per tile in the forward's launch order (longest lists first), one pixel per
// thread, 16x2 pixels per warp.  Batches of kBack terms are staged with the masks of the
// warps that may blend them, and each warp compacts a batch to its terms and walks them back
// to front, two per step: both weights before the two updates, one reduction for both.  A
// warp adds its sum of a term to the CTA's, or its few pixels one by one, and each
// (tile, Gaussian) slot is written once.  The sums' order is fixed within a warp and
// free among the warps.  Bound by instruction issue and the shared adds: 240 -> 181 us at
// 800x800 / 100k and 992 -> 769 at 1352x1014 / 300k against every term of a batch tested
// by every warp and reduced one at a time, in tile order.  Other orders of the same sums
// are faster, 111 and 536 us (8x4 pixels per warp, the opacity's factor multiplied into the
// sums, a place in shared memory per warp) and 129 and 626 (16x2 pixels and a place per
// warp), but a training step then sends plane cells the other way in 35 and 34 of 750
// steps of small and large scenes; here it is 23, where this order against itself has 20.
constexpr int kBack = 128;
constexpr int kFewPixels = 4;  // a warp adds up to this many pixels of a term one by one
constexpr int kBackWarps = kBatch / 32;

__global__ void __launch_bounds__(kBatch, 4) composite_bwd_kernel(const __grid_constant__ CompositeBwdArgs a) {
  __shared__ float s_acc[(kBack + 1) * kPairGrad];  // the terms' sums
  __shared__ float4 s_g0[kBack + 1];       // x, y, a2, c2 (the last place: a term that adds nothing)
  __shared__ float4 s_co[kBack + 1];       // conic, opacity
  __shared__ float4 s_col[kBack + 1];      // colour, b2
  __shared__ uint32_t s_slot[kBack], s_mask[kBack];
  __shared__ __align__(8) uint32_t s_list[kBackWarps][kBack];  // byte offsets of the warp's terms
  __shared__ int s_max_last;
  const int tile = a.order ? (int)a.order[blockIdx.x] : (int)blockIdx.x;
  const int tx = tile % a.tiles_x, ty = tile / a.tiles_x;
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const int px = tx * kTile + (int)(lane & 15), py = ty * kTile + (int)warp * 2 + (int)(lane >> 4);
  const bool inside = px < a.width && py < a.height;
  const int pix = py * a.width + px;
  const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
  const uint2 range = a.ranges[tile];
  const int n = (int)(range.y - range.x);
  const int last = inside ? a.n_contrib[pix] : 0;
  PixelBack p{1.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (inside) {
    p.T = a.t_final[pix];
    p.dC0 = a.dl_dimage[3 * pix];
    p.dC1 = a.dl_dimage[3 * pix + 1];
    p.dC2 = a.dl_dimage[3 * pix + 2];
  }
  if (threadIdx.x == 0) {
    s_max_last = 0;
    s_g0[kBack] = s_co[kBack] = s_col[kBack] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  const int wlast = __reduce_max_sync(0xffffffffu, last);
  if (lane == 0) atomicMax(&s_max_last, wlast);
  __syncthreads();
  const int max_last = min(s_max_last, n);
  const int term = (int)threadIdx.x % kBack, half = (int)threadIdx.x / kBack;

  for (int bstart = ((max_last - 1) / kBack) * kBack; bstart >= 0 && max_last > 0; bstart -= kBack) {
    __syncthreads();  // the previous batch's sums have been written out
    const int jend = min(kBack, max_last - bstart);
    for (int k = threadIdx.x; k < kBack * kPairGrad; k += kBatch) s_acc[k] = 0.f;
    if (term < jend) {
      const uint32_t g = a.values[range.x + bstart + term];
      const float4 co = a.conic_opacity[g];
      if (half == 0) {
        const float2 xy = a.xy[g];
        s_g0[term] = composite_coeffs(xy, co);
        s_co[term] = co;
        s_mask[term] = row_pair_mask(xy, co, composite_exp_threshold(co.w), tx, ty);
      } else {
        s_col[term] = make_float4(a.rgb[3 * (size_t)g], a.rgb[3 * (size_t)g + 1], a.rgb[3 * (size_t)g + 2],
                                  composite_b2(co));
        if (a.slot) {
          const int4 r = a.slot[g];
          s_slot[term] = (uint32_t)r.w + (uint32_t)((ty - r.y) * r.z + (tx - r.x));
        } else {
          const int4 r = a.rect[g];
          s_slot[term] = a.offsets[g] + (uint32_t)((ty - r.y) * (r.z - r.x) + (tx - r.x));
        }
      }
    }
    __syncthreads();
    int cnt = 0;
    for (int c0 = 0; c0 < jend; c0 += 32) {
      const int j = c0 + (int)lane;
      const bool hit = j < jend && ((s_mask[j] >> warp) & 1u);
      const uint32_t bal = __ballot_sync(0xffffffffu, hit);
      if (hit) s_list[warp][cnt + __popc(bal & ((1u << lane) - 1u))] = 16u * (uint32_t)j;
      cnt += __popc(bal);
    }
    if ((cnt & 1) && lane == 0) s_list[warp][cnt] = 16u * (uint32_t)kBack;
    __syncwarp();
    const int end = 16 * min(max(last - bstart, 0), kBack);  // byte offset past the pixel's last term
    for (int i = (cnt - 1) & ~1; i >= 0; i -= 2) {
      const uint2 l = *reinterpret_cast<const uint2*>(&s_list[warp][i]);  // l.y, the later one, first
      const float4 a0 = staged4(s_g0, l.y), b0 = staged4(s_g0, l.x), aco = staged4(s_co, l.y), bco = staged4(s_co, l.x);
      const float4 acol = staged4(s_col, l.y), bcol = staged4(s_col, l.x);
      const float2 ad = __fadd2_rn(make_float2(a0.x, a0.y), make_float2(-fx, -fy));
      const float2 bd = __fadd2_rn(make_float2(b0.x, b0.y), make_float2(-fx, -fy));
      float Ga, Gb;
      float alpha_a = composite_alpha(a0, acol.w, aco.w, ad.x, ad.y, Ga);
      float alpha_b = composite_alpha(b0, bcol.w, bco.w, bd.x, bd.y, Gb);
      if ((int)l.y >= end) alpha_a = 0.f;
      if ((int)l.x >= end) alpha_b = 0.f;
      // byte offset 16 j of term j is place (9/4) 16 j of its sums
      float* pa = reinterpret_cast<float*>(reinterpret_cast<char*>(s_acc) + (l.y >> 2) * kPairGrad);
      float* pb = reinterpret_cast<float*>(reinterpret_cast<char*>(s_acc) + (l.x >> 2) * kPairGrad);
      const unsigned ma = __ballot_sync(0xffffffffu, alpha_a > 0.f), mb = __ballot_sync(0xffffffffu, alpha_b > 0.f);
      if ((ma | mb) == 0u) continue;
      float ga[kPairGrad], gb[kPairGrad], s8;
      term_grads(p, alpha_a, Ga, aco, acol, ad.x, ad.y, ga);
      term_grads(p, alpha_b, Gb, bco, bcol, bd.x, bd.y, gb);
      const bool many_a = __popc(ma) > kFewPixels, many_b = __popc(mb) > kFewPixels;
      if (many_a || many_b) {
        const float s = warp_sum18(ga, gb, lane, s8);
        const bool last = (lane & 15u) == 1u;  // (value 8 from the first odd lane)
        if ((lane < 16 ? many_a : many_b) && ((lane & 1u) == 0u || last))
          atomicAdd((lane < 16 ? pa : pb) + (last ? 8 : (lane >> 1) & 7u), last ? s8 : s);
      }
      if (!many_a && alpha_a > 0.f)
#pragma unroll
        for (int k = 0; k < kPairGrad; ++k) atomicAdd(&pa[k], ga[k]);
      if (!many_b && alpha_b > 0.f)
#pragma unroll
        for (int k = 0; k < kPairGrad; ++k) atomicAdd(&pb[k], gb[k]);
    }
    __syncthreads();
    if (term < jend) {  // half 0: values 0..3 of the term, half 1: values 4..8
      const float* v = s_acc + term * kPairGrad + 4 * half;
      float4* dst = reinterpret_cast<float4*>(a.grad_pair + (size_t)s_slot[term] * kPairStride);
      dst[half] = make_float4(v[0], v[1], v[2], v[3]);
      if (half) dst[2] = make_float4(v[4], 0.f, 0.f, 0.f);
    }
  }
}

// ------------------------------------------------------------------ projection

// Real SH basis and its derivative with respect to the direction components,
// differentiating the same formulas the forward evaluates.
constexpr float kY00 = 0.28209479177387814f, kY1 = 0.48860251190291992f, kY2a = 1.0925484305920792f,
                kY20 = 0.31539156525252005f, kY22 = 0.54627421529603959f, kY33 = 0.59004358992664352f,
                kY32 = 2.8906114426405538f, kY31 = 0.45704579946446572f, kY30 = 0.37317633259011540f,
                kY32b = 1.4453057213202769f;

__device__ void sh_basis_and_grad(int deg, float x, float y, float z, float* Y, float (*dY)[3]) {
#pragma unroll
  for (int k = 0; k < 16; ++k) Y[k] = dY[k][0] = dY[k][1] = dY[k][2] = 0.f;
  Y[0] = kY00;
  if (deg < 1) return;
  Y[1] = kY1 * y; Y[2] = kY1 * z; Y[3] = kY1 * x;
  dY[1][1] = kY1; dY[2][2] = kY1; dY[3][0] = kY1;
  if (deg < 2) return;
  const float xx = x * x, yy = y * y, zz = z * z;
  Y[4] = kY2a * x * y; dY[4][0] = kY2a * y; dY[4][1] = kY2a * x;
  Y[5] = kY2a * y * z; dY[5][1] = kY2a * z; dY[5][2] = kY2a * y;
  Y[6] = kY20 * (3.f * zz - 1.f); dY[6][2] = 6.f * kY20 * z;
  Y[7] = kY2a * x * z; dY[7][0] = kY2a * z; dY[7][2] = kY2a * x;
  Y[8] = kY22 * (xx - yy); dY[8][0] = 2.f * kY22 * x; dY[8][1] = -2.f * kY22 * y;
  if (deg < 3) return;
  Y[9] = kY33 * y * (3.f * xx - yy); dY[9][0] = 6.f * kY33 * x * y; dY[9][1] = kY33 * (3.f * xx - 3.f * yy);
  Y[10] = kY32 * x * y * z; dY[10][0] = kY32 * y * z; dY[10][1] = kY32 * x * z; dY[10][2] = kY32 * x * y;
  Y[11] = kY31 * y * (5.f * zz - 1.f); dY[11][1] = kY31 * (5.f * zz - 1.f); dY[11][2] = 10.f * kY31 * y * z;
  Y[12] = kY30 * z * (5.f * zz - 3.f); dY[12][2] = kY30 * (15.f * zz - 3.f);
  Y[13] = kY31 * x * (5.f * zz - 1.f); dY[13][0] = kY31 * (5.f * zz - 1.f); dY[13][2] = 10.f * kY31 * x * z;
  Y[14] = kY32b * z * (xx - yy); dY[14][0] = 2.f * kY32b * x * z; dY[14][1] = -2.f * kY32b * y * z;
  dY[14][2] = kY32b * (xx - yy);
  Y[15] = kY33 * x * (xx - 3.f * yy); dY[15][0] = kY33 * (3.f * xx - 3.f * yy); dY[15][1] = -6.f * kY33 * x * y;
}

// The SH colour's backward for one Gaussian with K coefficients per channel at `row` (its
// coefficients, which its dL/dSH replaces), and the gradient with respect to the view
// direction.
template <int K>
__device__ __forceinline__ void sh_colour_bwd(float* row, const float (&Y)[16], const float (&dY)[16][3],
                                              const float (&G9)[kPairGrad], float& gdir0, float& gdir1,
                                              float& gdir2) {
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) {
    float raw = 0.5f, shv[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      shv[k] = row[3 * k + ch];
      raw += Y[k] * shv[k];
    }
    const bool live = raw > 0.f;  // clamped at 0: no gradient
    const float gr = live ? G9[6 + ch] : 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      row[3 * k + ch] = gr * Y[k];
      const float s = gr * shv[k];
      gdir0 += s * dY[k][0];
      gdir1 += s * dY[k][1];
      gdir2 += s * dY[k][2];
    }
  }
}

// One Gaussian from the sums of its slots (g9) and its SH row, which dL/dSH replaces.
template <int K>
__device__ __forceinline__ void project_bwd_gaussian(const ProjectBwdArgs& a, int g, const float* g9, float* sh_row) {
  if (g >= a.n) return;
  float* gd = a.gd + 10 * (size_t)g;
  if (a.radius[g] == 0) {
#pragma unroll
    for (int k = 0; k < 10; ++k) gd[k] = 0.f;
#pragma unroll
    for (int k = 0; k < 3 * K; ++k) sh_row[k] = 0.f;
    return;
  }
  float G9[kPairGrad];
#pragma unroll
  for (int k = 0; k < kPairGrad; ++k) G9[k] = g9[k];
  if (a.stat_grad) {  // densification statistics: view-space gradient norm of the visible Gaussian
    a.stat_grad[g] += sqrtf(G9[0] * G9[0] + G9[1] * G9[1]);
    a.stat_visible[g] += 1.f;
  }
  const CamParams& c = a.cam;
  const float4 co = a.conic_opacity[g];
  if (a.g_opacity) a.g_opacity[g] += G9[5] * co.w * (1.f - co.w);

  const float X0 = a.means[3 * g], X1 = a.means[3 * g + 1], X2 = a.means[3 * g + 2];
  float gX0 = 0.f, gX1 = 0.f, gX2 = 0.f;
  // ---- SH colour
  {
    const float cpx = -(c.m[0] * c.m[3] + c.m[4] * c.m[7] + c.m[8] * c.m[11]);
    const float cpy = -(c.m[1] * c.m[3] + c.m[5] * c.m[7] + c.m[9] * c.m[11]);
    const float cpz = -(c.m[2] * c.m[3] + c.m[6] * c.m[7] + c.m[10] * c.m[11]);
    const float vx = X0 - cpx, vy = X1 - cpy, vz = X2 - cpz;
    const float vn = sqrtf(vx * vx + vy * vy + vz * vz), vinv = 1.f / vn;
    const float dx = vx * vinv, dy = vy * vinv, dz = vz * vinv;
    float Y[16], dY[16][3];
    sh_basis_and_grad(K == 1 ? 0 : K == 4 ? 1 : K == 9 ? 2 : 3, dx, dy, dz, Y, dY);
    float gdir0 = 0.f, gdir1 = 0.f, gdir2 = 0.f;
    sh_colour_bwd<K>(sh_row, Y, dY, G9, gdir0, gdir1, gdir2);
    const float dd = dx * gdir0 + dy * gdir1 + dz * gdir2;
    gX0 += (gdir0 - dx * dd) * vinv;
    gX1 += (gdir1 - dy * dd) * vinv;
    gX2 += (gdir2 - dz * dd) * vinv;
  }
  // ---- camera-space mean and the projected mean
  const float px = c.m[0] * X0 + c.m[1] * X1 + c.m[2] * X2 + c.m[3];
  const float py = c.m[4] * X0 + c.m[5] * X1 + c.m[6] * X2 + c.m[7];
  const float pz = c.m[8] * X0 + c.m[9] * X1 + c.m[10] * X2 + c.m[11];
  const float iz = 1.f / pz, iz2 = iz * iz;
  float gp0 = G9[0] * c.fx * iz, gp1 = G9[1] * c.fy * iz;
  float gp2 = -G9[0] * c.fx * px * iz2 - G9[1] * c.fy * py * iz2;
  // ---- conic = Sigma2D^-1: dL/dSigma2D = -K G_K K
  const float ka = co.x, kb = co.y, kc = co.z;
  const float gka = G9[2], gkb = 0.5f * G9[3], gkc = G9[4];
  // M = K G_K, then -M K
  const float m00 = ka * gka + kb * gkb, m01 = ka * gkb + kb * gkc;
  const float m10 = kb * gka + kc * gkb, m11 = kb * gkb + kc * gkc;
  const float S00 = -(m00 * ka + m01 * kb), S01 = -(m00 * kb + m01 * kc);
  const float S10 = -(m10 * ka + m11 * kb), S11 = -(m10 * kb + m11 * kc);
  // ---- Sigma2D = A A^T + 0.3 I, A = T R S, T = J W
  const float4 q4 = reinterpret_cast<const float4*>(a.quats)[g];
  const float qn = sqrtf(q4.x * q4.x + q4.y * q4.y + q4.z * q4.z + q4.w * q4.w), qinv = 1.f / qn;
  const float w = q4.x * qinv, x = q4.y * qinv, y = q4.z * qinv, z = q4.w * qinv;
  float R[3][3] = {{1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y)},
                   {2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x)},
                   {2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)}};
  const float sc[3] = {expf(a.log_scales[3 * g]), expf(a.log_scales[3 * g + 1]), expf(a.log_scales[3 * g + 2])};
  const float limx = kGuard * (float)c.guard_w / (2.f * c.fx), limy = kGuard * (float)c.guard_h / (2.f * c.fy);
  const float rx_raw = px * iz, ry_raw = py * iz;
  const bool clx = fabsf(rx_raw) > limx, cly = fabsf(ry_raw) > limy;
  const float rx = fminf(limx, fmaxf(-limx, rx_raw)), ry = fminf(limy, fmaxf(-limy, ry_raw));
  const float J00 = c.fx * iz, J02 = -c.fx * rx * iz, J11 = c.fy * iz, J12 = -c.fy * ry * iz;
  float T[2][3] = {{J00 * c.m[0] + J02 * c.m[8], J00 * c.m[1] + J02 * c.m[9], J00 * c.m[2] + J02 * c.m[10]},
                   {J11 * c.m[4] + J12 * c.m[8], J11 * c.m[5] + J12 * c.m[9], J11 * c.m[6] + J12 * c.m[10]}};
  float RS[3][3], A[2][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) RS[i][j] = R[i][j] * sc[j];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) A[i][j] = T[i][0] * RS[0][j] + T[i][1] * RS[1][j] + T[i][2] * RS[2][j];
  // dL/dA = (S + S^T) A
  const float Ss00 = 2.f * S00, Ss01 = S01 + S10, Ss11 = 2.f * S11;
  float gA[2][3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    gA[0][j] = Ss00 * A[0][j] + Ss01 * A[1][j];
    gA[1][j] = Ss01 * A[0][j] + Ss11 * A[1][j];
  }
  float gT[2][3], gRS[3][3];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) gT[i][j] = gA[i][0] * RS[j][0] + gA[i][1] * RS[j][1] + gA[i][2] * RS[j][2];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) gRS[i][j] = T[0][i] * gA[0][j] + T[1][i] * gA[1][j];
  float gR[3][3], gsc[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      gR[i][j] = gRS[i][j] * sc[j];
      gsc[j] += gRS[i][j] * R[i][j];
    }
  // dR/dq for the unit quaternion (w, x, y, z)
  const float gw = 2.f * (-z * gR[0][1] + y * gR[0][2] + z * gR[1][0] - x * gR[1][2] - y * gR[2][0] + x * gR[2][1]);
  const float gx = 2.f * (y * gR[0][1] + z * gR[0][2] + y * gR[1][0] - w * gR[1][2] + z * gR[2][0] + w * gR[2][1]) -
                   4.f * x * (gR[1][1] + gR[2][2]);
  const float gy = 2.f * (x * gR[0][1] + w * gR[0][2] + x * gR[1][0] + z * gR[1][2] - w * gR[2][0] + z * gR[2][1]) -
                   4.f * y * (gR[0][0] + gR[2][2]);
  const float gz = 2.f * (-w * gR[0][1] + x * gR[0][2] + w * gR[1][0] + y * gR[1][2] + x * gR[2][0] + y * gR[2][1]) -
                   4.f * z * (gR[0][0] + gR[1][1]);
  const float qd = w * gw + x * gx + y * gy + z * gz;
  // T = J W: dL/dJ = dL/dT W^T (only the non-zero entries of J matter)
  const float gJ00 = gT[0][0] * c.m[0] + gT[0][1] * c.m[1] + gT[0][2] * c.m[2];
  const float gJ02 = gT[0][0] * c.m[8] + gT[0][1] * c.m[9] + gT[0][2] * c.m[10];
  const float gJ11 = gT[1][0] * c.m[4] + gT[1][1] * c.m[5] + gT[1][2] * c.m[6];
  const float gJ12 = gT[1][0] * c.m[8] + gT[1][1] * c.m[9] + gT[1][2] * c.m[10];
  gp2 += -gJ00 * c.fx * iz2 - gJ11 * c.fy * iz2;
  if (!clx) {
    gp0 += -gJ02 * c.fx * iz2;
    gp2 += gJ02 * 2.f * c.fx * px * iz2 * iz;
  } else {
    gp2 += gJ02 * c.fx * rx * iz2;
  }
  if (!cly) {
    gp1 += -gJ12 * c.fy * iz2;
    gp2 += gJ12 * 2.f * c.fy * py * iz2 * iz;
  } else {
    gp2 += gJ12 * c.fy * ry * iz2;
  }
  gX0 += c.m[0] * gp0 + c.m[4] * gp1 + c.m[8] * gp2;
  gX1 += c.m[1] * gp0 + c.m[5] * gp1 + c.m[9] * gp2;
  gX2 += c.m[2] * gp0 + c.m[6] * gp1 + c.m[10] * gp2;
  const float gq[4] = {(gw - w * qd) * qinv, (gx - x * qd) * qinv, (gy - y * qd) * qinv, (gz - z * qd) * qinv};
  const float gs[3] = {gsc[0] * sc[0], gsc[1] * sc[1], gsc[2] * sc[2]};
  gd[0] = gX0; gd[1] = gX1; gd[2] = gX2;
  gd[3] = gq[0]; gd[4] = gq[1]; gd[5] = gq[2]; gd[6] = gq[3];
  gd[7] = gs[0]; gd[8] = gs[1]; gd[9] = gs[2];
  if (a.g_means) {
    a.g_means[3 * g] += gX0; a.g_means[3 * g + 1] += gX1; a.g_means[3 * g + 2] += gX2;
  }
  if (a.g_quats)
#pragma unroll
    for (int k = 0; k < 4; ++k) a.g_quats[4 * g + k] += gq[k];
  if (a.g_log_scales)
#pragma unroll
    for (int k = 0; k < 3; ++k) a.g_log_scales[3 * g + k] += gs[k];
}

// 128 Gaussians per CTA.  Their SH rows come into shared memory as one block (16-byte
// copies, in flight while the slots are summed) and their gradients leave it the same way;
// the slots of a Gaussian are summed by four lanes, one per 16 bytes of a slot, with four
// slots in flight.  One thread per Gaussian reading its own rows and slots waited for
// scattered 16-byte accesses: 177 against 148 us for 300k Gaussians of degree 3, 55 against
// 48 for 100k.
constexpr int kProj = 128;
template <int K>
__global__ void __launch_bounds__(kProj) project_bwd_kernel(const __grid_constant__ ProjectBwdArgs a) {
  constexpr int F = 3 * K, FS = F % 2 ? F : F % 4 ? F + 1 : F + 4;  // row stride: odd, or 16-byte rows 4 banks on
  constexpr bool kVec = F % 4 == 0;
  __shared__ __align__(16) float s_sh[kProj * FS];
  __shared__ float s_g9[kProj][13];
  const int g0 = blockIdx.x * kProj, g = g0 + (int)threadIdx.x, m = min(kProj, a.n - g0);
  if (kVec) {
    for (int e = threadIdx.x; e < m * (F / 4); e += kProj) {
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_sh + (e / (F / 4)) * FS + 4 * (e % (F / 4)));
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst),
                   "l"(reinterpret_cast<const float4*>(a.sh + (size_t)g0 * F) + e)
                   : "memory");
    }
  } else {
    for (int e = threadIdx.x; e < m * F; e += kProj) s_sh[(e / F) * FS + e % F] = a.sh[(size_t)g0 * F + e];
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  // the pair slots (contiguous per Gaussian by construction)
  const int part = threadIdx.x & 3;
#pragma unroll 1
  for (int q = threadIdx.x >> 2; q < m; q += kProj / 4) {
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    if (part < 3 && a.radius[g0 + q] != 0) {
      const int4 rc = a.rect[g0 + q];
      const uint32_t cnt = (uint32_t)((rc.z - rc.x) * (rc.w - rc.y));
      const float4* src = reinterpret_cast<const float4*>(a.grad_pair + (size_t)a.offsets[g0 + q] * kPairStride) + part;
      constexpr int kU = 4;
      for (uint32_t e = 0; e < cnt; e += kU) {
        float4 v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
          v[u] = e + u < cnt ? src[(size_t)(e + u) * (kPairStride / 4)] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          sum.x += v[u].x; sum.y += v[u].y; sum.z += v[u].z; sum.w += v[u].w;
        }
      }
    }
    if (part < 3) {
      float* dst = &s_g9[q][4 * part];
      dst[0] = sum.x;
      if (part < 2) {
        dst[1] = sum.y; dst[2] = sum.z; dst[3] = sum.w;
      }
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  project_bwd_gaussian<K>(a, g, s_g9[threadIdx.x], s_sh + threadIdx.x * FS);
  if (!a.g_sh) return;
  __syncthreads();  // every row holds dL/dSH
  if (kVec) {
    for (int e = threadIdx.x; e < m * (F / 4); e += kProj) {
      float4* out = reinterpret_cast<float4*>(a.g_sh + (size_t)g0 * F) + e;
      const float4 v = *reinterpret_cast<const float4*>(s_sh + (e / (F / 4)) * FS + 4 * (e % (F / 4)));
      float4 o = *out;
      o.x += v.x; o.y += v.y; o.z += v.z; o.w += v.w;
      *out = o;
    }
  } else {
    for (int e = threadIdx.x; e < m * F; e += kProj) a.g_sh[(size_t)g0 * F + e] += s_sh[(e / F) * FS + e % F];
  }
}

}  // namespace

cudaError_t launch_composite_bwd(const CompositeBwdArgs& a, cudaStream_t s) {
  const int tiles_y = (a.height + kTile - 1) / kTile;
  if (a.tiles_x * tiles_y == 0) return cudaSuccess;
  composite_bwd_kernel<<<a.tiles_x * tiles_y, kBatch, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_project_bwd(const ProjectBwdArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)((a.n + kProj - 1) / kProj);
  switch (a.sh_degree) {
    case 0: project_bwd_kernel<1><<<grid, kProj, 0, s>>>(a); break;
    case 1: project_bwd_kernel<4><<<grid, kProj, 0, s>>>(a); break;
    case 2: project_bwd_kernel<9><<<grid, kProj, 0, s>>>(a); break;
    case 3: project_bwd_kernel<16><<<grid, kProj, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace fs4d
