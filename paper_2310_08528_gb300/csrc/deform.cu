// Gaussian deformation field, float32 SIMT path (Sec. 4.2, Eq. 5, Eq. 6).
//
// Persistent CTAs (one per SM) of one or two independent groups of 256 threads, each
// walking tiles of TG Gaussians of its own behind named barriers.  Per tile:
//   1. Eq. 5: normalise (x, y, z) by the scene box and t to [-1, 1], bilinearly
//      interpolate the six planes xy xz yz xt yt zt of every level and multiply
//      them channel-wise.  h/4 consecutive lanes share one (Gaussian, level) item
//      and each owns one float4 of features, so a warp's loads cover whole grid
//      vertices (channels-last) with many requests in flight per thread;
//   2. phi_d (two ReLU layers) and the three heads as register-blocked SIMT
//      GEMMs: thread (warp w, lane l) computes outputs 8w..8w+7 of TG/32 consecutive
//      Gaussians, so with TG = 128 one 128-bit activation load and two broadcast 128-bit
//      weight loads feed 32 FMAs.  Every output keeps the order b + sum_i w_i x_i of a
//      plain dot product;
//   3. Eq. 6: add the deltas to X, r, s, each thread for the outputs that it summed.
// Activations live feature-major in shared memory ([feature][TG + 4]: the padding keeps
// both access patterns conflict-free); the MLP is kept transposed (Wt[in][out]) and
// shared by the groups.
//
// Bound by the FP32 FMAs (21.1k per Gaussian) and, with one group of eight warps, by
// their latency: a group's plane taps, barriers and output layers left the FMA pipe
// idle.  Two groups fill it for each other: 417 -> 348 us for the 300k room (343 with
// the layers unrolled by eight; its FMAs alone take 157), now at 73% of the shared-memory and L1 data pipe (a k-step of a warp costs
// four wavefronts for its activations and two for each weight load).
// While every tile of 32 can run at once, a call takes those: more SMs share the chain of a
// tile (2000 Gaussians 24.1 -> 15.0 us, 5000 32.4 -> 25.4, 9000 25.5; in two rounds, at 19,000,
// they take 44 us and tiles of 128 take 33).
#include "fs4d_internal.cuh"

namespace fs4d {
namespace {


__device__ __forceinline__ void axis_setup(float u, int R, int& i0, float& f) {
  const float uc = fminf(1.f, fmaxf(-1.f, u));
  const float g = (uc + 1.f) * 0.5f * (float)(R - 1);
  int i = (int)floorf(g);
  i = max(0, min(i, R - 2));
  i0 = i;
  f = g - (float)i;
}

constexpr int kThreads = 256;        // threads of a group

// MLP floats for HL input features (MlpGeomT::total: padded to a multiple of 4)
constexpr int mlp_floats(int hl) {
  return (hl * kWidth + kWidth + 4 * (kWidth * kWidth + kWidth) + kDeltaDim * (kWidth + 1) + 3) / 4 * 4;
}

// Shared memory of a CTA: the weights, then per group the activations X [max(HL, 64)][TG + 4]
// and Hd [64][TG + 4] and the rows (X, t).
constexpr size_t smem_bytes(int hl, int tg, int groups) {
  return 4 * (size_t)mlp_floats(hl) +
         (size_t)groups * (4 * (size_t)((hl > kWidth ? hl : kWidth) + kWidth) * (tg + 4) + 16 * (size_t)tg);
}

__device__ __forceinline__ void group_bar(int grp) { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(kThreads)); }

// acc[g][o] = b[o8 + o] + sum_i Wt[i][o8 + o] * src[i][g0 + g], in input order.
template <int IN, int TG>
__device__ __forceinline__ void layer64(const float* __restrict__ Wt, const float* __restrict__ b,
                                        const float* __restrict__ src, int g0, int o8, float (&acc)[TG / 32][8]) {
  constexpr int GP = TG / 32, kGS = TG + 4;
  // outputs in pairs: one f32x2 FMA per two outputs (each element the same FP32 FMA)
  float2 a2[GP][4];
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    const float2 bo = make_float2(b[o8 + 2 * o], b[o8 + 2 * o + 1]);
#pragma unroll
    for (int g = 0; g < GP; ++g) a2[g][o] = bo;
  }
#pragma unroll 8
  for (int i = 0; i < IN; ++i) {
    float xs[GP];
    if constexpr (GP == 4) {
      const float4 x = *reinterpret_cast<const float4*>(src + i * kGS + g0);
      xs[0] = x.x; xs[1] = x.y; xs[2] = x.z; xs[3] = x.w;
    } else if constexpr (GP == 2) {
      const float2 x = *reinterpret_cast<const float2*>(src + i * kGS + g0);
      xs[0] = x.x; xs[1] = x.y;
    } else {
      xs[0] = src[i * kGS + g0];
    }
    const float4 w0 = *reinterpret_cast<const float4*>(Wt + i * kWidth + o8);
    const float4 w1 = *reinterpret_cast<const float4*>(Wt + i * kWidth + o8 + 4);
    const float2 ws[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                          make_float2(w1.z, w1.w)};
#pragma unroll
    for (int g = 0; g < GP; ++g) {
      const float2 xg = make_float2(xs[g], xs[g]);
#pragma unroll
      for (int o = 0; o < 4; ++o) a2[g][o] = __ffma2_rn(ws[o], xg, a2[g][o]);
    }
  }
#pragma unroll
  for (int g = 0; g < GP; ++g)
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      acc[g][2 * o] = a2[g][o].x;
      acc[g][2 * o + 1] = a2[g][o].y;
    }
}

template <int TG>
__device__ __forceinline__ void store_relu(float* __restrict__ dst, int g0, int o8, const float (&acc)[TG / 32][8]) {
  constexpr int GP = TG / 32, kGS = TG + 4;
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    float* d = dst + (o8 + o) * kGS + g0;
    if constexpr (GP == 4)
      *reinterpret_cast<float4*>(d) =
          make_float4(fmaxf(acc[0][o], 0.f), fmaxf(acc[1][o], 0.f), fmaxf(acc[2][o], 0.f), fmaxf(acc[3][o], 0.f));
    else
#pragma unroll
      for (int g = 0; g < GP; ++g) d[g] = fmaxf(acc[g][o], 0.f);
  }
}

// Output layer of one head for Gaussian g, outputs j0 .. j0 + NPS - 1 (those below OUT):
// d[k] = b2[j] + sum_o W2[o][j] * hid[o][g].
template <int OUT, int NPS, int TG>
__device__ __forceinline__ void head_out(const float* __restrict__ W2, const float* __restrict__ b2,
                                         const float* __restrict__ hid, int g, int j0, float (&d)[NPS]) {
  constexpr int kGS = TG + 4;
  int j[NPS];
#pragma unroll
  for (int k = 0; k < NPS; ++k) {
    j[k] = min(j0 + k, OUT - 1);  // (an output past the last is summed and not used)
    d[k] = b2[j[k]];
  }
#pragma unroll 8
  for (int o = 0; o < kWidth; ++o) {
    const float x = hid[o * kGS + g];
#pragma unroll
    for (int k = 0; k < NPS; ++k) d[k] = fmaf(W2[o * OUT + j[k]], x, d[k]);
  }
}

// The recompute for the backward: the thread's activations (after ReLU) as rows of out and
// a bit for each that is positive.
template <int TG>
__device__ __forceinline__ void put_acts(const float (&acc)[TG / 32][8], int o8, float* __restrict__ out, int ld,
                                         long long row0, long long n, uint32_t* mask_word) {
  uint32_t mask = 0;
#pragma unroll
  for (int g = 0; g < TG / 32; ++g) {
    float v[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      v[o] = fmaxf(acc[g][o], 0.f);
      mask |= v[o] > 0.f ? 1u << (8 * g + o) : 0u;
    }
    if (row0 + g < n) {
      float4* q = reinterpret_cast<float4*>(out + (row0 + g) * ld + o8);
      q[0] = make_float4(v[0], v[1], v[2], v[3]);
      q[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
  }
  *mask_word = mask;
}

// ACT: the backward's recompute (DeformArgs::act_masks).
template <int H, int L, int TG, int GROUPS, bool ACT>
__global__ void __launch_bounds__(GROUPS * kThreads, 1) deform_fp32_kernel(const __grid_constant__ DeformArgs a) {
  constexpr int HL = H * L;
  constexpr int XR = HL > kWidth ? HL : kWidth;
  constexpr int Q = H / 4;  // float4 groups per grid vertex
  constexpr int kGS = TG + 4;
  constexpr int SLOTS = kThreads / TG;       // threads per Gaussian
  constexpr int NPS = (4 + SLOTS - 1) / SLOTS;  // outputs of a head per thread
  extern __shared__ float4 smem4[];
  const int grp = threadIdx.x / kThreads, gt = threadIdx.x % kThreads;
  float* sw = reinterpret_cast<float*>(smem4);
  float* X = sw + mlp_floats(HL) + (size_t)grp * (XR + kWidth) * kGS;   // [XR][kGS]: f_h, then a1, then f_d (in place)
  float* Hd = X + XR * kGS;                                             // [64][kGS]: hidden layer of the current head
  float4* sRowX = reinterpret_cast<float4*>(sw + mlp_floats(HL) + (size_t)GROUPS * (XR + kWidth) * kGS) + grp * TG;
  // the weights by cp.async (every 16-byte copy in flight at once), waited for
  // before the first tile's MLP below
  for (int i = threadIdx.x; i < a.mg.total / 4; i += GROUPS * kThreads) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem4 + i);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(reinterpret_cast<const float4*>(a.mlp_t) + i)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  // the weights above are the scene's; the rows below may come from earlier work
  pdl_wait();
  pdl_trigger();
  for (long long i = (long long)blockIdx.x * GROUPS * kThreads + threadIdx.x; i < a.zero_n16;
       i += (long long)gridDim.x * GROUPS * kThreads)
    a.zero[i] = make_uint4(0u, 0u, 0u, 0u);

  const int warp = gt >> 5, lane = gt & 31;
  const int g0 = lane * (TG / 32), o8 = warp * 8;
  const int myg = gt % TG, j0 = (gt / TG) * NPS;  // this thread's Gaussian and first output of each head
  const PlaneGeom& pg = a.pg;
  const MlpGeomT& mg = a.mg;
  const long long total = (long long)a.n * a.n_t;
  const long long tiles = (total + TG - 1) / TG;
  bool loaded = false;
  // (the first groups of all CTAs before the second ones)
  for (long long tile = blockIdx.x + (long long)gridDim.x * grp; tile < tiles; tile += (long long)gridDim.x * GROUPS) {
    const long long base = tile * TG;
    // ---- 0. the tile's rows (the work-order index, then position, t, quaternion and
    // log-scales in one round of loads): the position into shared memory, and what Eq. 6
    // adds to, with this thread's outputs
    float bm[NPS], bq[NPS], bs[NPS];
    int g = 0, ti = 0;
    {
      const long long gi = base + myg;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < NPS; ++k) bm[k] = bq[k] = bs[k] = 0.f;
      if (gi < total) {
        ti = (int)(gi / a.n);
        const int gw = (int)(gi - (long long)ti * a.n);
        g = a.perm ? (int)a.perm[gw] : gw;  // spatially coherent work order
        x = make_float4(a.means[3 * (size_t)g], a.means[3 * (size_t)g + 1], a.means[3 * (size_t)g + 2],
                        a.ts ? a.ts[ti] : a.t0);
#pragma unroll
        for (int k = 0; k < NPS; ++k) {
          if (j0 + k < 4) bq[k] = a.quats[4 * (size_t)g + j0 + k];
          if (j0 + k < 3) {
            bm[k] = a.means[3 * (size_t)g + j0 + k];
            bs[k] = a.log_scales[3 * (size_t)g + j0 + k];
          }
        }
      }
      if (gt < TG) sRowX[gt] = x;  // (last read while the previous tile was sampled)
    }
    group_bar(grp);
    // ---- 1. Eq. 5 into X[0..HL)
    for (int item = gt; item < TG * L * Q; item += kThreads) {
      const int q = item % Q, rl = item / Q;
      const int r = rl % TG, l = rl / TG;
      const long long gi = base + r;
      float f[4] = {0.f, 0.f, 0.f, 0.f};
      if (gi < total) {
        const float4 xr = sRowX[r];
        float c[4];
        c[0] = (xr.x - pg.aabb_min[0]) * pg.aabb_scale[0] - 1.f;
        c[1] = (xr.y - pg.aabb_min[1]) * pg.aabb_scale[1] - 1.f;
        c[2] = (xr.z - pg.aabb_min[2]) * pg.aabb_scale[2] - 1.f;
        c[3] = 2.f * xr.w - 1.f;
        f[0] = f[1] = f[2] = f[3] = 1.f;
#pragma unroll
        for (int p = 0; p < 6; ++p) {
          const int ax = (p < 2) ? 0 : (p == 2 ? 1 : p - 3);  // xy xz yz xt yt zt
          const int bx = (p == 0) ? 1 : (p <= 2 ? 2 : 3);
          const int Ra = ax < 3 ? pg.res[l] : pg.res_time;
          const int Rb = bx < 3 ? pg.res[l] : pg.res_time;
          int i0, jj;
          float fa, fb;
          axis_setup(c[ax], Ra, i0, fa);
          axis_setup(c[bx], Rb, jj, fb);
          const float4* v00 =
              reinterpret_cast<const float4*>(a.planes + pg.off[l][p] + ((long long)jj * Ra + i0) * H) + q;
          const float4 A = __ldg(v00), B = __ldg(v00 + Q), C = __ldg(v00 + (long long)Ra * Q),
                       E = __ldg(v00 + (long long)Ra * Q + Q);
          const float w00 = (1.f - fa) * (1.f - fb), w10 = fa * (1.f - fb), w01 = (1.f - fa) * fb, w11 = fa * fb;
          f[0] *= w00 * A.x + w10 * B.x + w01 * C.x + w11 * E.x;
          f[1] *= w00 * A.y + w10 * B.y + w01 * C.y + w11 * E.y;
          f[2] *= w00 * A.z + w10 * B.z + w01 * C.z + w11 * E.z;
          f[3] *= w00 * A.w + w10 * B.w + w01 * C.w + w11 * E.w;
        }
      }
      // rows 4q..4q+3 of column r; the store order is rotated by q/2 so that the
      // lanes of one store hit 32 distinct banks
      float* dst = X + (l * H + 4 * q) * kGS + r;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int e = (s + (q >> 1)) & 3;
        const float v = e == 0 ? f[0] : (e == 1 ? f[1] : (e == 2 ? f[2] : f[3]));
        dst[e * kGS] = v;
      }
      if (ACT && gi < total)
        *reinterpret_cast<float4*>(a.act_fh + gi * HL + l * H + 4 * q) = make_float4(f[0], f[1], f[2], f[3]);
    }
    if (!loaded) {  // every thread takes part in this barrier once, here or after the loop
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      __syncthreads();
      loaded = true;
    } else {
      group_bar(grp);
    }
    // ---- 2. phi_d, in place in X
    float acc[TG / 32][8];
    layer64<HL, TG>(sw + mg.w[0], sw + mg.b[0], X, g0, o8, acc);
    group_bar(grp);
    store_relu<TG>(X, g0, o8, acc);
    uint32_t* masks = ACT ? a.act_masks + tile * 5 * kThreads + gt : nullptr;
    if (ACT) put_acts<TG>(acc, o8, a.act_a1, kWidth, base + g0, total, masks);
    group_bar(grp);
    layer64<kWidth, TG>(sw + mg.w[1], sw + mg.b[1], X, g0, o8, acc);
    group_bar(grp);
    store_relu<TG>(X, g0, o8, acc);
    if constexpr (ACT) {
      put_acts<TG>(acc, o8, a.fd_out, kWidth, base + g0, total, masks + kThreads);
      group_bar(grp);
#pragma unroll
      for (int h = 0; h < 3; ++h) {
        layer64<kWidth, TG>(sw + mg.w[2 + 2 * h], sw + mg.b[2 + 2 * h], X, g0, o8, acc);
        put_acts<TG>(acc, o8, a.act_hid + kWidth * h, 3 * kWidth, base + g0, total, masks + (2 + h) * kThreads);
      }
      continue;  // (the next tile writes X after a barrier)
    }
    group_bar(grp);
    if (a.fd_out) {  // f_d for the colour and opacity heads, rows in work order
      for (int e = gt; e < TG * kWidth; e += kThreads) {
        const int r = e / kWidth, k = e - r * kWidth;
        if (base + r < total) a.fd_out[(size_t)(base + r) * kWidth + k] = X[k * kGS + r];
      }
    }
    // heads phi_x, phi_r, phi_s: hidden layer into Hd, then the output layer; ---- 3. Eq. 6
    const bool live = base + myg < total;
    const long long o = a.out_tab ? (long long)g : (long long)ti * a.n + g;
    float d[NPS];
    layer64<kWidth, TG>(sw + mg.w[2], sw + mg.b[2], X, g0, o8, acc);
    store_relu<TG>(Hd, g0, o8, acc);  // (its last readers are a barrier or more behind)
    group_bar(grp);
    if (j0 < 3) {
      head_out<3, NPS, TG>(sw + mg.w[3], sw + mg.b[3], Hd, myg, j0, d);
      float* om = a.out_tab ? a.out_tab[3 * ti] : a.out_means;
#pragma unroll
      for (int k = 0; k < NPS; ++k)
        if (live && j0 + k < 3) om[3 * o + j0 + k] = bm[k] + d[k];
    }
    layer64<kWidth, TG>(sw + mg.w[4], sw + mg.b[4], X, g0, o8, acc);
    group_bar(grp);
    store_relu<TG>(Hd, g0, o8, acc);
    group_bar(grp);
    if (j0 < 4) {
      head_out<4, NPS, TG>(sw + mg.w[5], sw + mg.b[5], Hd, myg, j0, d);
      float* oq = a.out_tab ? a.out_tab[3 * ti + 1] : a.out_quats;
#pragma unroll
      for (int k = 0; k < NPS; ++k)
        if (live && j0 + k < 4) oq[4 * o + j0 + k] = bq[k] + d[k];
    }
    layer64<kWidth, TG>(sw + mg.w[6], sw + mg.b[6], X, g0, o8, acc);
    group_bar(grp);
    store_relu<TG>(Hd, g0, o8, acc);
    group_bar(grp);
    if (j0 < 3) {
      head_out<3, NPS, TG>(sw + mg.w[7], sw + mg.b[7], Hd, myg, j0, d);
      float* os = a.out_tab ? a.out_tab[3 * ti + 2] : a.out_log_scales;
#pragma unroll
      for (int k = 0; k < NPS; ++k)
        if (live && j0 + k < 3) os[3 * o + j0 + k] = bs[k] + d[k];
    }
  }
  if (!loaded) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
  }
}

template <int H, int L, int TG, int GROUPS, bool ACT>
cudaError_t launch_tg(const DeformArgs& a, cudaStream_t s) {
  constexpr size_t smem = smem_bytes(H * L, TG, GROUPS);
  static_assert(smem <= 227 * 1024, "one CTA's shared memory");
  if (a.mg.total != mlp_floats(H * L)) return cudaErrorInvalidValue;
  static PerDeviceFlag attr;
  cudaError_t e = once_per_device(attr, [&] {
    return cudaFuncSetAttribute(deform_fp32_kernel<H, L, TG, GROUPS, ACT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem);
  });
  if (e != cudaSuccess) return e;
  const int sms = device_sm_count();
  const long long total = (long long)a.n * a.n_t;
  const long long need = (total + TG - 1) / TG;
  const int grid = (int)(need < sms ? need : sms);
  return launch_kernel(!a.mlp_late, deform_fp32_kernel<H, L, TG, GROUPS, ACT>, dim3((unsigned)grid), GROUPS * kThreads, smem, s, a);
}

template <int H, int L>
cudaError_t launch_t(const DeformArgs& a, cudaStream_t s) {
  // two groups where their activations fit beside the weights (up to 64 input features)
  constexpr int kGroups = smem_bytes(H * L, 128, 2) <= 227 * 1024 ? 2 : 1;
  const long long total = (long long)a.n * a.n_t;
  // tiles of 32 while all of them run at once
  if (a.act_masks) return launch_tg<H, L, 128, kGroups, true>(a, s);
  if (total <= 64ll * device_sm_count()) return launch_tg<H, L, 32, 2, false>(a, s);
  return launch_tg<H, L, 128, kGroups, false>(a, s);
}

}  // namespace

bool deform_fp32_supported(int feat_dim, int n_levels) {
  return (feat_dim == 16 || feat_dim == 32) && n_levels >= 1 && n_levels <= 3;
}

cudaError_t launch_deform_fp32(const DeformArgs& a, cudaStream_t s) {
  if ((long long)a.n * a.n_t == 0) return cudaSuccess;
  const int h = a.pg.feat_dim, L = a.pg.n_levels;
  if (h == 16 && L == 1) return launch_t<16, 1>(a, s);
  if (h == 16 && L == 2) return launch_t<16, 2>(a, s);
  if (h == 16 && L == 3) return launch_t<16, 3>(a, s);
  if (h == 32 && L == 1) return launch_t<32, 1>(a, s);
  if (h == 32 && L == 2) return launch_t<32, 2>(a, s);
  if (h == 32 && L == 3) return launch_t<32, 3>(a, s);
  return cudaErrorInvalidValue;
}

}  // namespace fs4d
