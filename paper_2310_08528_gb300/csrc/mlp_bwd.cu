// Backward of the deformation (Sec. 4.2, Eq. 5, Eq. 6): the heads, phi_d, the HexPlane
// sampling and the weight gradients, in float32.  Four steps over the Gaussians in the
// scene's work order, with every activation and delta that a weight gradient reads as a
// row per Gaussian ([n][features]):
//   1. the forward is recomputed by the float32 deformation kernel (deform.cu), the same
//      sums in the same order, which leaves the activations and one bit per ReLU;
//   2. mlp_delta_kernel: the chain of transposed layers, 128 Gaussians per group of 256
//      threads, two groups per CTA, register-blocked as the forward;
//   3. plane_bwd_kernel: the plane cells (128-bit float atomics: many Gaussians share a
//      cell) and the sampling positions;
//   4. wgrad kernels: dW = D^T X as 8x8 register blocks per thread, per-chunk partial sums
//      and a fixed-order reduction (deterministic).
// 100k Gaussians, L = 2, h = 32: recompute, deltas and planes 457 us, weights 133; one
// kernel for all but the weights took 635, the weights 244.
#include <algorithm>

#include "fs4d_internal.cuh"

namespace fs4d {
namespace {

constexpr int kThreads = 256;   // threads of a group
constexpr int kGroups = 2;
constexpr int kTG = 128;        // Gaussians per tile
constexpr int kGS = kTG + 4;    // row stride of the shared delta array

__device__ __forceinline__ void group_bar(int grp) { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(kThreads)); }

// Floats of the layers a CTA keeps, as [out][in]: the three head hidden layers, d2, d1 and
// the ten rows of the output layers.
template <int HL>
constexpr int delta_weights() {
  return 4 * kWidth * kWidth + kWidth * HL + kDeltaDim * kWidth;
}

// acc[g][i8 + i] += sum_o D[o][g0 + g] W[o][i8 + i] over 64 outputs o.
template <int LDW>
__device__ __forceinline__ void back64(const float* __restrict__ W, const float* __restrict__ D, int g0, int i8,
                                       float2 (&acc)[4][4]) {
#pragma unroll 8
  for (int o = 0; o < kWidth; ++o) {
    const float4 x = *reinterpret_cast<const float4*>(D + o * kGS + g0);
    const float4 w0 = *reinterpret_cast<const float4*>(W + o * LDW + i8);
    const float4 w1 = *reinterpret_cast<const float4*>(W + o * LDW + i8 + 4);
    const float xs[4] = {x.x, x.y, x.z, x.w};
    const float2 ws[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                          make_float2(w1.z, w1.w)};
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const float2 xg = make_float2(xs[g], xs[g]);
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[g][k] = __ffma2_rn(ws[k], xg, acc[g][k]);
    }
  }
}

__device__ __forceinline__ void clear(float2 (&acc)[4][4]) {
#pragma unroll
  for (int g = 0; g < 4; ++g)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[g][k] = make_float2(0.f, 0.f);
}

// The thread's 4 x 8 deltas with the ReLU mask applied (bit 8 g + o), into shared memory
// [o][g] and as rows of `out`.
__device__ __forceinline__ void put_deltas(float2 (&acc)[4][4], uint32_t mask, float* __restrict__ D, int g0, int o8,
                                           float* __restrict__ out, int ld, long long row0, long long n) {
  float v[4][8];
#pragma unroll
  for (int g = 0; g < 4; ++g)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[g][2 * k] = (mask >> (8 * g + 2 * k)) & 1u ? acc[g][k].x : 0.f;
      v[g][2 * k + 1] = (mask >> (8 * g + 2 * k + 1)) & 1u ? acc[g][k].y : 0.f;
    }
#pragma unroll
  for (int o = 0; o < 8; ++o)
    *reinterpret_cast<float4*>(D + (o8 + o) * kGS + g0) = make_float4(v[0][o], v[1][o], v[2][o], v[3][o]);
#pragma unroll
  for (int g = 0; g < 4; ++g)
    if (row0 + g < n) {
      float4* q = reinterpret_cast<float4*>(out + (row0 + g) * ld + o8);
      q[0] = make_float4(v[g][0], v[g][1], v[g][2], v[g][3]);
      q[1] = make_float4(v[g][4], v[g][5], v[g][6], v[g][7]);
    }
}

// Bound by the FMAs and the shared-memory reads that feed them, as the forward.
template <int HL>
__global__ void __launch_bounds__(kGroups * kThreads, 1) mlp_delta_kernel(const __grid_constant__ MlpBwdArgs a) {
  extern __shared__ float4 smem4[];
  const int grp = threadIdx.x / kThreads, gt = threadIdx.x % kThreads;
  float* sw = reinterpret_cast<float*>(smem4);
  const float* Wh = sw;                                   // [3][64][64]
  const float* W2 = sw + 3 * kWidth * kWidth;             // [64][64]
  const float* W1 = sw + 4 * kWidth * kWidth;             // [64][HL]
  const float* Wo = W1 + kWidth * HL;                     // [10][64]
  float* D = sw + delta_weights<HL>() + grp * (kWidth + kDeltaDim) * kGS;  // [64][kGS]: a layer's deltas
  float* DO = D + kWidth * kGS;                                            // [10][kGS]: dL/d(X', r', s')
  {  // the layers from the source layout (W then b of d1 d2 x1 x2 r1 r2 s1 s2)
    const int in1 = kWidth * HL + kWidth, sq = kWidth * kWidth + kWidth;
    const int outs[3] = {3, 4, 3}, col0[3] = {0, 3, 7};
    int off = in1 + sq;
    auto copy = [&](float* dst, int src, int count) {
      for (int i = threadIdx.x; i < count; i += kGroups * kThreads) dst[i] = __ldg(a.mlp + src + i);
    };
    copy(sw + 4 * kWidth * kWidth, 0, kWidth * HL);
    copy(sw + 3 * kWidth * kWidth, in1, kWidth * kWidth);
    for (int h = 0; h < 3; ++h) {
      copy(sw + h * kWidth * kWidth, off, kWidth * kWidth);
      off += sq;
      copy(sw + 4 * kWidth * kWidth + kWidth * HL + col0[h] * kWidth, off, outs[h] * kWidth);
      off += outs[h] * kWidth + outs[h];
    }
  }
  __syncthreads();
  const int warp = gt >> 5, lane = gt & 31;
  const int g0 = 4 * lane, o8 = 8 * warp;
  const long long n = a.f.n, tiles = (n + kTG - 1) / kTG;
  for (long long tile = blockIdx.x + (long long)gridDim.x * grp; tile < tiles; tile += (long long)gridDim.x * kGroups) {
    const long long base = tile * kTG, row0 = base + g0;
    uint32_t mask[5];  // a1, f_d, the heads' hidden layers
#pragma unroll
    for (int k = 0; k < 5; ++k) mask[k] = a.f.act_masks[(tile * 5 + k) * kThreads + gt];
    if (gt < kTG) {
      float v[12] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (base + gt < n) {
        const long long g = a.f.perm ? (long long)a.f.perm[base + gt] : base + gt;
#pragma unroll
        for (int j = 0; j < kDeltaDim; ++j) v[j] = a.gd[kDeltaDim * g + j];
        float4* q = reinterpret_cast<float4*>(a.act.dout + 12 * (base + gt));
#pragma unroll
        for (int j = 0; j < 3; ++j) q[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      }
#pragma unroll
      for (int j = 0; j < kDeltaDim; ++j) DO[j * kGS + gt] = v[j];
    }
    group_bar(grp);
    float2 fd[4][4], d[4][4];
    clear(fd);
#pragma unroll
    for (int h = 0; h < 3; ++h) {
      // d_hid = ReLU'(hid) W_out^T dL/d(X', r', s')
      constexpr int kOuts[3] = {3, 4, 3}, kCol0[3] = {0, 3, 7};
      clear(d);
#pragma unroll
      for (int j = 0; j < kOuts[h]; ++j) {
        const float4 x = *reinterpret_cast<const float4*>(DO + (kCol0[h] + j) * kGS + g0);
        const float4 w0 = *reinterpret_cast<const float4*>(Wo + (kCol0[h] + j) * kWidth + o8);
        const float4 w1 = *reinterpret_cast<const float4*>(Wo + (kCol0[h] + j) * kWidth + o8 + 4);
        const float xs[4] = {x.x, x.y, x.z, x.w};
        const float2 ws[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                              make_float2(w1.z, w1.w)};
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
          for (int k = 0; k < 4; ++k) d[g][k] = __ffma2_rn(ws[k], make_float2(xs[g], xs[g]), d[g][k]);
      }
      if (h > 0) group_bar(grp);  // the previous head's deltas have been read
      put_deltas(d, mask[2 + h], D, g0, o8, a.act.dh + kWidth * h, 3 * kWidth, row0, n);
      group_bar(grp);
      back64<kWidth>(Wh + h * kWidth * kWidth, D, g0, o8, fd);
    }
    group_bar(grp);
    put_deltas(fd, mask[1], D, g0, o8, a.act.d2, kWidth, row0, n);
    group_bar(grp);
    clear(d);
    back64<kWidth>(W2, D, g0, o8, d);
    group_bar(grp);
    put_deltas(d, mask[0], D, g0, o8, a.act.d1, kWidth, row0, n);
    group_bar(grp);
    // dL/df_h, 64 features per pass
#pragma unroll
    for (int i0 = 0; i0 < HL; i0 += kWidth) {
      if (i0 + o8 < HL) {
        clear(d);
        back64<HL>(W1 + i0, D, g0, o8, d);
#pragma unroll
        for (int g = 0; g < 4; ++g)
          if (row0 + g < n) {
            float4* q = reinterpret_cast<float4*>(a.act.dfh + (row0 + g) * HL + i0 + o8);
            q[0] = make_float4(d[g][0].x, d[g][0].y, d[g][1].x, d[g][1].y);
            q[1] = make_float4(d[g][2].x, d[g][2].y, d[g][3].x, d[g][3].y);
          }
      }
    }
    group_bar(grp);  // (the next tile writes DO and D)
  }
}

// ------------------------------------------------------------------ HexPlane

__device__ __forceinline__ void axis_setup(float u, int R, int& i0, float& f, float& dfdu) {
  const float uc = fminf(1.f, fmaxf(-1.f, u));
  const float g = (uc + 1.f) * 0.5f * (float)(R - 1);
  int i = (int)floorf(g);
  i = max(0, min(i, R - 2));
  i0 = i;
  f = g - (float)i;
  dfdu = (u > -1.f && u < 1.f) ? 0.5f * (float)(R - 1) : 0.f;
}

// h/4 consecutive lanes per Gaussian, a float4 of features each, level after level (so a
// Gaussian's position gradient is one lane's sum, level by level, and needs no atomics).  All Gaussians
// share t, so a time plane's gradient falls on two lines of cells, the two time rows: the
// atomics go to kTimeCopies copies of them (by CTA, against many adds to one address),
// which time_lines_kernel adds up.  300k Gaussians with the recompute and the deltas: 1398
// us straight into the planes, 1186 with eight copies (1194 with the positions level by
// level, as their adds to memory were), 1263 with two; three CTAs per SM
// instead of two 1198.  One line per axis that the two rows' weights multiply at the end
// took half the adds (1097), but the products' other rounding turned the sign of a sum near
// zero, and with it Adam's step, for 17 seeds of 30 against 1 for either form above.
constexpr int kTimeCopies = 8;
template <int H, int L>
__global__ void __launch_bounds__(256, 2) plane_bwd_kernel(const __grid_constant__ MlpBwdArgs a) {
  constexpr int Q = H / 4, HL = H * L;
  const DeformArgs& f = a.f;
  const PlaneGeom& pg = f.pg;
  const long long item = (long long)blockIdx.x * 256 + threadIdx.x;
  const int q = (int)(item % Q);
  const long long ii = item / Q;
  const bool live = ii < f.n;
  const long long g = live ? (f.perm ? (long long)f.perm[ii] : ii) : 0;
  float c[4] = {0.f, 0.f, 0.f, 2.f * f.t0 - 1.f}, gm[3] = {0.f, 0.f, 0.f};
  if (live)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      c[k] = (f.means[3 * g + k] - pg.aabb_min[k]) * pg.aabb_scale[k] - 1.f;
      if (a.g_means && q == 0) gm[k] = a.g_means[3 * g + k];
    }
  int line0 = 0;  // first cell of the level in a line
#pragma unroll 1
  for (int l = 0; l < L; line0 += pg.res[l], ++l) {
    float gxs[3] = {0.f, 0.f, 0.f};
    if (live) {
      const float4 gf4 = *reinterpret_cast<const float4*>(a.act.dfh + ii * HL + l * H + 4 * q);
      const float gf[4] = {gf4.x, gf4.y, gf4.z, gf4.w};
      int i0[4];
      float fr[4], df[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) axis_setup(c[k], k < 3 ? pg.res[l] : pg.res_time, i0[k], fr[k], df[k]);
      float v[6][4];
#pragma unroll
      for (int p = 0; p < 6; ++p) {
        const int ax = (p < 2) ? 0 : (p == 2 ? 1 : p - 3), bx = (p == 0) ? 1 : (p <= 2 ? 2 : 3);
        const int Ra = ax < 3 ? pg.res[l] : pg.res_time;
        const float4* v00 =
            reinterpret_cast<const float4*>(f.planes + pg.off[l][p] + ((long long)i0[bx] * Ra + i0[ax]) * H) + q;
        const float4 A = __ldg(v00), B = __ldg(v00 + Q), C = __ldg(v00 + (long long)Ra * Q),
                     E = __ldg(v00 + (long long)Ra * Q + Q);
        const float fa = fr[ax], fb = fr[bx];
        const float w00 = (1.f - fa) * (1.f - fb), w10 = fa * (1.f - fb), w01 = (1.f - fa) * fb, w11 = fa * fb;
        v[p][0] = w00 * A.x + w10 * B.x + w01 * C.x + w11 * E.x;
        v[p][1] = w00 * A.y + w10 * B.y + w01 * C.y + w11 * E.y;
        v[p][2] = w00 * A.z + w10 * B.z + w01 * C.z + w11 * E.z;
        v[p][3] = w00 * A.w + w10 * B.w + w01 * C.w + w11 * E.w;
      }
#pragma unroll
      for (int p = 0; p < 6; ++p) {
        const int ax = (p < 2) ? 0 : (p == 2 ? 1 : p - 3), bx = (p == 0) ? 1 : (p <= 2 ? 2 : 3);
        const int Ra = ax < 3 ? pg.res[l] : pg.res_time;
        float gv[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float others = 1.f;
#pragma unroll
          for (int r = 0; r < 6; ++r)
            if (r != p) others *= v[r][e];
          gv[e] = gf[e] * others;
        }
        const long long cell = pg.off[l][p] + ((long long)i0[bx] * Ra + i0[ax]) * H + 4 * q;
        const float* P = f.planes + cell;
        const float4 A = __ldg(reinterpret_cast<const float4*>(P)), B = __ldg(reinterpret_cast<const float4*>(P + H)),
                     C = __ldg(reinterpret_cast<const float4*>(P + (long long)Ra * H)),
                     E = __ldg(reinterpret_cast<const float4*>(P + (long long)Ra * H + H));
        const float fa = fr[ax], fb = fr[bx];
        const float As[4] = {A.x, A.y, A.z, A.w}, Bs[4] = {B.x, B.y, B.z, B.w}, Cs[4] = {C.x, C.y, C.z, C.w},
                    Es[4] = {E.x, E.y, E.z, E.w};
        float sa = 0.f, sb = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          sa += gv[e] * ((1.f - fb) * (Bs[e] - As[e]) + fb * (Es[e] - Cs[e]));
          sb += gv[e] * ((1.f - fa) * (Cs[e] - As[e]) + fa * (Es[e] - Bs[e]));
        }
        if (a.g_planes) {
          float* GP = a.g_planes + cell;
          long long up = (long long)Ra * H;  // to the next row of the second axis
          if (p >= 3) {
            up = 3ll * a.act.line_cells * H;
            GP = a.act.lines + (((long long)(blockIdx.x % kTimeCopies) * 6 + ax) * a.act.line_cells + line0 + i0[ax]) * H + 4 * q;
          }
          const float w00 = (1.f - fa) * (1.f - fb), w10 = fa * (1.f - fb), w01 = (1.f - fa) * fb, w11 = fa * fb;
          atomicAdd(reinterpret_cast<float4*>(GP), make_float4(w00 * gv[0], w00 * gv[1], w00 * gv[2], w00 * gv[3]));
          atomicAdd(reinterpret_cast<float4*>(GP + H),
                    make_float4(w10 * gv[0], w10 * gv[1], w10 * gv[2], w10 * gv[3]));
          atomicAdd(reinterpret_cast<float4*>(GP + up),
                    make_float4(w01 * gv[0], w01 * gv[1], w01 * gv[2], w01 * gv[3]));
          atomicAdd(reinterpret_cast<float4*>(GP + up + H),
                    make_float4(w11 * gv[0], w11 * gv[1], w11 * gv[2], w11 * gv[3]));
        }
        if (ax < 3) gxs[ax] += sa * df[ax] * pg.aabb_scale[ax];
        if (bx < 3) gxs[bx] += sb * df[bx] * pg.aabb_scale[bx];
      }
    }
    // the level's position gradient: the Q lanes of one Gaussian are consecutive and Q divides 32
    if (!a.g_means) continue;
#pragma unroll
    for (int w = 1; w < Q; w <<= 1)
#pragma unroll
      for (int k = 0; k < 3; ++k) gxs[k] += __shfl_xor_sync(0xffffffffu, gxs[k], w);
#pragma unroll
    for (int k = 0; k < 3; ++k) gm[k] += gxs[k];
  }
  if (a.g_means && live && q == 0)
#pragma unroll
    for (int k = 0; k < 3; ++k) a.g_means[3 * g + k] = gm[k];
}

// The lines of the time planes (all copies) into their two time rows.
__global__ void __launch_bounds__(256) time_lines_kernel(const __grid_constant__ MlpBwdArgs a) {
  const PlaneGeom& pg = a.f.pg;
  const int H = pg.feat_dim;
  const int e = blockIdx.x * 256 + (int)threadIdx.x, per = a.act.line_cells * H;
  if (e >= 3 * per) return;
  const int ax = e / per;
  int cell = (e % per) / H, l = 0;
  float g0 = 0.f, g1 = 0.f;
#pragma unroll
  for (int k = 0; k < kTimeCopies; ++k) {
    g0 += a.act.lines[(long long)(2 * k) * 3 * per + e];
    g1 += a.act.lines[(long long)(2 * k + 1) * 3 * per + e];
  }
  for (; cell >= pg.res[l]; ++l) cell -= pg.res[l];
  int j0;
  float fb, db;
  axis_setup(2.f * a.f.t0 - 1.f, pg.res_time, j0, fb, db);
  float* out = a.g_planes + pg.off[l][3 + ax] + ((long long)j0 * pg.res[l] + cell) * H + e % H;
  out[0] += g0;
  out[(long long)pg.res[l] * H] += g1;
}

// ------------------------------------------------------------------ weight gradients

constexpr int kWChunk = 512;   // Gaussians per partial sum
constexpr int kWStage = 64;    // Gaussians staged per step, in four slices of 16

// Partial sums over one chunk of Gaussians of dW[o][i] = sum_n D[n][o] X[n][i] and
// db[o] = sum_n D[n][o].  Each slice of 64 threads holds a whole 64 x 64 block, 8 x 8 per
// thread (rows 4 ob .. and 32 + 4 ob .., columns alike, so that the 16-byte shared reads of
// a warp are consecutive), and takes a quarter of the staged Gaussians: four reads feed 64
// FMAs.  The slices are added up in a fixed order.  The output layers (O <= 4 rows) take a
// column per thread.
constexpr size_t kWSmem = 4 * 2 * 2 * (size_t)kWStage * kWidth;
__global__ void __launch_bounds__(256, 2) wgrad_partial_kernel(const __grid_constant__ WgradArgs wa) {
  extern __shared__ float4 smem4[];
  __shared__ float s_bias[4][kWidth];
  float* sD = reinterpret_cast<float*>(smem4);            // [2][kWStage][64]
  float* sX = sD + 2 * kWStage * kWidth;                  // [2][kWStage][64]
  const WgradLayer& ly = wa.l[blockIdx.y];
  const int O = ly.O, I = ly.I;
  const bool wide = O > 4;
  const long long n0 = (long long)blockIdx.x * kWChunk, n1 = min(wa.n, n0 + kWChunk);
  const int slice = threadIdx.x >> 6, t = threadIdx.x & 63;
  const int ib = t & 7, ob = t >> 3;
  auto stage = [&](int buf, long long b0) {
    float* d = sD + buf * kWStage * kWidth;
    float* x = sX + buf * kWStage * kWidth;
    auto async16 = [](float* dst, const float* src) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                   : "memory");
    };
    for (int e = threadIdx.x; e < kWStage * kWidth / 4; e += 256) {
      const int r = e / (kWidth / 4), c = 4 * (e % (kWidth / 4));
      const bool row = b0 + r < n1;
      if (row && c < I)
        async16(x + r * kWidth + c, ly.X + (b0 + r) * ly.ldx + c);
      else
        *reinterpret_cast<float4*>(x + r * kWidth + c) = make_float4(0.f, 0.f, 0.f, 0.f);
      if (!wide) continue;
      if (row)
        async16(d + r * kWidth + c, ly.D + (b0 + r) * ly.ldd + c);
      else
        *reinterpret_cast<float4*>(d + r * kWidth + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (!wide)  // four rows of deltas (the ones past O are another head's and are not used)
      for (int e = threadIdx.x; e < kWStage * 4; e += 256)
        d[e] = b0 + e / 4 < n1 && e % 4 < O ? ly.D[(b0 + e / 4) * ly.ldd + e % 4] : 0.f;
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  float2 acc[8][4];
  float bias = 0.f;
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[r][k] = make_float2(0.f, 0.f);
  const int brow = ib < 4 ? 4 * ob + ib : 32 + 4 * ob + ib - 4;  // the row whose bias this thread sums
  stage(0, n0);
  int buf = 0;
  for (long long b0 = n0; b0 < n1; b0 += kWStage, buf ^= 1) {
    if (b0 + kWStage < n1) {
      stage(buf ^ 1, b0 + kWStage);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    const float* d = sD + buf * kWStage * kWidth;
    const float* x = sX + buf * kWStage * kWidth;
    if (wide) {
#pragma unroll 2
      for (int j = 16 * slice; j < 16 * slice + 16; ++j) {
        const float4 d0 = *reinterpret_cast<const float4*>(d + j * kWidth + 4 * ob);
        const float4 d1 = *reinterpret_cast<const float4*>(d + j * kWidth + 32 + 4 * ob);
        const float4 x0 = *reinterpret_cast<const float4*>(x + j * kWidth + 4 * ib);
        const float4 x1 = *reinterpret_cast<const float4*>(x + j * kWidth + 32 + 4 * ib);
        bias += d[j * kWidth + brow];
        const float dv[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
        const float2 xv[4] = {make_float2(x0.x, x0.y), make_float2(x0.z, x0.w), make_float2(x1.x, x1.y),
                              make_float2(x1.z, x1.w)};
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float2 dr = make_float2(dv[r], dv[r]);
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[r][k] = __ffma2_rn(dr, xv[k], acc[r][k]);
        }
      }
    } else {
      for (int j = 16 * slice; j < 16 * slice + 16; ++j) {
        const float4 d4 = *reinterpret_cast<const float4*>(d + 4 * j);
        const float2 xx = make_float2(x[j * kWidth + t], x[j * kWidth + t]);
        acc[0][0] = __ffma2_rn(make_float2(d4.x, d4.y), xx, acc[0][0]);
        acc[0][1] = __ffma2_rn(make_float2(d4.z, d4.w), xx, acc[0][1]);
        if (t < 4) bias += d[4 * j + t];
      }
    }
    __syncthreads();  // this buffer is refilled by the next step
  }
  // the slices' sums through shared memory: [slice][64][64]
  float* red = reinterpret_cast<float*>(smem4) + slice * kWidth * kWidth;
  if (wide) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int o = r < 4 ? 4 * ob + r : 32 + 4 * ob + r - 4;
      *reinterpret_cast<float4*>(red + o * kWidth + 4 * ib) =
          make_float4(acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
      *reinterpret_cast<float4*>(red + o * kWidth + 32 + 4 * ib) =
          make_float4(acc[r][2].x, acc[r][2].y, acc[r][3].x, acc[r][3].y);
    }
    s_bias[slice][brow] = bias;
  } else {
    red[t] = acc[0][0].x;
    red[kWidth + t] = acc[0][0].y;
    red[2 * kWidth + t] = acc[0][1].x;
    red[3 * kWidth + t] = acc[0][1].y;
    if (t < 4) s_bias[slice][t] = bias;
  }
  __syncthreads();
  const float* all = reinterpret_cast<const float*>(smem4);
  float* partial = wa.partial + ly.part_off + (long long)blockIdx.x * (O * I + O);
  for (int e = threadIdx.x; e < O * kWidth; e += 256) {
    const int o = e / kWidth, i = e % kWidth;
    const float s = (all[e] + all[e + kWidth * kWidth]) + (all[e + 2 * kWidth * kWidth] + all[e + 3 * kWidth * kWidth]);
    if (i < I) partial[o * I + i] = s;
  }
  if ((int)threadIdx.x < O) {
    const int o = threadIdx.x;
    partial[O * I + o] = (s_bias[0][o] + s_bias[1][o]) + (s_bias[2][o] + s_bias[3][o]);
  }
}

// Four threads per weight (adjacent lanes), each summing every fourth chunk in
// eight running sums (eight loads in flight), then the four combined by two
// shuffles: a fixed order, so the result is deterministic.
constexpr int kRedSplit = 4;
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const __grid_constant__ WgradArgs wa) {
  const WgradLayer& ly = wa.l[blockIdx.y];
  const int O = ly.O, I = ly.I;
  const int E = O * I + O;
  const int e = blockIdx.x * (blockDim.x / kRedSplit) + (int)threadIdx.x / kRedSplit;
  const int split = (int)threadIdx.x % kRedSplit;
  const bool live = e < E;  // (every lane stays for the shuffles)
  const float* partial = wa.partial + ly.part_off;
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (live) {
    int c = split, k = 0;
    for (; c + 7 * kRedSplit < wa.chunks; c += 8 * kRedSplit) {
#pragma unroll
      for (int u = 0; u < 8; ++u) acc[u] += partial[(long long)(c + u * kRedSplit) * E + e];
    }
    for (; c < wa.chunks; c += kRedSplit, ++k) acc[k & 7] += partial[(long long)c * E + e];
  }
  float s = ((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7]));
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  if (!live || split != 0) return;
  if (e < O * I)
    ly.gW[(long long)(e / I) * ly.ldw + e % I] += s;
  else if (ly.gb)
    ly.gb[e - O * I] += s;
}

template <int H, int L>
cudaError_t launch_bwd_t(const MlpBwdArgs& a, cudaStream_t s) {
  constexpr int HL = H * L;
  constexpr size_t smem = 4 * ((size_t)delta_weights<HL>() + (size_t)kGroups * (kWidth + kDeltaDim) * kGS);
  static_assert(smem <= 227 * 1024, "one CTA's shared memory");
  static PerDeviceFlag attr;
  cudaError_t e = once_per_device(attr, [&] {
    return cudaFuncSetAttribute(mlp_delta_kernel<HL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (e != cudaSuccess) return e;
  const long long tiles = ((long long)a.f.n + kTG - 1) / kTG;
  const int sms = device_sm_count();
  mlp_delta_kernel<HL><<<(unsigned)(tiles < sms ? tiles : sms), kGroups * kThreads, smem, s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t line_floats = 3 * (size_t)a.act.line_cells * H;
  if (a.g_planes && (e = cudaMemsetAsync(a.act.lines, 0, 4 * 2 * kTimeCopies * line_floats, s)) != cudaSuccess) return e;
  const long long items = (long long)a.f.n * (H / 4);
  plane_bwd_kernel<H, L><<<(unsigned)((items + 255) / 256), 256, 0, s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess || !a.g_planes) return e;
  time_lines_kernel<<<(unsigned)((line_floats + 255) / 256), 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

namespace {
int line_cells(const PlaneGeom& pg) {
  int c = 0;
  for (int l = 0; l < pg.n_levels; ++l) c += pg.res[l];
  return c;
}
}  // namespace

size_t mlp_act_floats(long long n, const PlaneGeom& pg) {
  const long long tiles = (n + kTG - 1) / kTG;
  return (size_t)n * (2 * pg.feat_dim * pg.n_levels + 64 + 64 + 192 + 12 + 192 + 64 + 64) +
         (size_t)tiles * 5 * kThreads + (size_t)kTimeCopies * 6 * line_cells(pg) * pg.feat_dim;
}

MlpActs mlp_acts(float* base, long long n, const PlaneGeom& pg) {
  MlpActs q{};
  const int hin = pg.feat_dim * pg.n_levels;
  const long long tiles = (n + kTG - 1) / kTG;
  auto take = [&](long long w) {
    float* p = base;
    base += n * w;
    return p;
  };
  q.fh = take(hin); q.a1 = take(64); q.fd = take(64); q.hid = take(192); q.dout = take(12);
  q.dh = take(192); q.d2 = take(64); q.d1 = take(64); q.dfh = take(hin);
  q.masks = reinterpret_cast<uint32_t*>(base);
  q.lines = base + tiles * 5 * kThreads;
  q.line_cells = line_cells(pg);
  return q;
}

cudaError_t launch_mlp_bwd(const MlpBwdArgs& args, cudaStream_t s) {
  if (args.f.n <= 0) return cudaSuccess;
  MlpBwdArgs a = args;
  a.f.act_fh = a.act.fh; a.f.act_a1 = a.act.a1; a.f.fd_out = a.act.fd; a.f.act_hid = a.act.hid;
  a.f.act_masks = a.act.masks;
  const cudaError_t e = launch_deform_fp32(a.f, s);
  if (e != cudaSuccess) return e;
  const int h = a.f.pg.feat_dim, L = a.f.pg.n_levels;
  if (h == 16 && L == 1) return launch_bwd_t<16, 1>(a, s);
  if (h == 16 && L == 2) return launch_bwd_t<16, 2>(a, s);
  if (h == 16 && L == 3) return launch_bwd_t<16, 3>(a, s);
  if (h == 32 && L == 1) return launch_bwd_t<32, 1>(a, s);
  if (h == 32 && L == 2) return launch_bwd_t<32, 2>(a, s);
  if (h == 32 && L == 3) return launch_bwd_t<32, 3>(a, s);
  return cudaErrorInvalidValue;
}

long long wgrad_chunks(long long n) { return (n + kWChunk - 1) / kWChunk; }

cudaError_t launch_wgrad(WgradArgs& a, cudaStream_t s) {
  if (a.n <= 0 || a.n_layers <= 0) return cudaSuccess;
  a.chunks = (int)wgrad_chunks(a.n);
  int maxE = 0;
  long long off = 0;
  for (int k = 0; k < a.n_layers; ++k) {
    const WgradLayer& l = a.l[k];
    if (l.O > 64 || (l.O > 4 && l.O != 64) || l.I > 64 || (l.I & 3)) return cudaErrorInvalidValue;
    const int E = l.O * l.I + l.O;
    a.l[k].part_off = off;
    off += (long long)a.chunks * E;
    maxE = std::max(maxE, E);
  }
  static PerDeviceFlag attr;
  cudaError_t e = once_per_device(attr, [] {
    return cudaFuncSetAttribute(wgrad_partial_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWSmem);
  });
  if (e != cudaSuccess) return e;
  wgrad_partial_kernel<<<dim3(a.chunks, a.n_layers), 256, kWSmem, s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  wgrad_reduce_kernel<<<dim3((maxE + 256 / kRedSplit - 1) / (256 / kRedSplit), a.n_layers), 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace fs4d
