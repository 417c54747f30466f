// closure.cu - learned closure: dataset generation, training and inference
// entry points (kernels for the network itself live in closure.cuh).
//
// Training data are made by the solver: a fine periodic dense run is
// box-filtered by r^3 (mean populations), the filtered populations are
// streamed one coarse step (what a coarse voxel pulls) and turned into
// features; the target is the least-squares eddy viscosity over each coarse
// voxel's 3^3 neighbourhood, d_tau = 3 nu_t with
// nu_t = - sum tau_sgs_dev : S / sum 2 rho S : S,
// tau_sgs = mean(rho u u) - rho u_bar u_bar and S the central-difference strain
// of u_bar, clamped to [-(tau_c - 1/2) + 1e-3, 1/2].
// Training is plain FP32 on CUDA cores (the batch GEMMs are small): forward,
// backward, Adam, deterministic loop orders; minibatches are drawn with the
// SplitMix64 generator (Steele, Lea and Flood, OOPSLA 2014) on the counter
// step * batch + b.
#include <cmath>
#include <vector>

#include "closure.cuh"
#include "d3q19.cuh"
#include "exact.cuh"
#include "grid.h"

namespace lbm {

// parameter offsets in the flat FP32 vector
constexpr int P_W1 = 0, P_B1 = 1024, P_W2 = 1088, P_B2 = 5184, P_W3 = 5248, P_B3 = 5312;

// ------------------------------------------------------------ inference checks

__global__ void __launch_bounds__(256) k_mlp_forward_bf16(const ClosureParams* p, const float* X,
                                                          int64_t n, float* y) {
  __shared__ ClosureSmem sm;
  __shared__ __nv_bfloat16 stage[8][32 * FSTAGE];
  closure_load_smem(sm, p);
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  float x[MLP_IN];
#pragma unroll
  for (int k = 0; k < MLP_IN; ++k) x[k] = i < n ? X[i * MLP_IN + k] : 0.f;
  const float out = mlp_bf16_warp(x, sm, stage[threadIdx.x >> 5]);
  if (i < n) y[i] = out;
}

__global__ void k_mlp_forward_fp32(const float* th, const float* X, int64_t n, float* y) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float x[MLP_IN], h1[MLP_H];
  for (int k = 0; k < MLP_IN; ++k) x[k] = X[i * MLP_IN + k];
  for (int j = 0; j < MLP_H; ++j) {
    float z = th[P_B1 + j];
    for (int k = 0; k < MLP_IN; ++k) z += th[P_W1 + j * MLP_IN + k] * x[k];
    h1[j] = fmaxf(z, 0.f);
  }
  float out = th[P_B3];
  for (int j = 0; j < MLP_H; ++j) {
    float z = th[P_B2 + j];
    for (int k = 0; k < MLP_H; ++k) z += th[P_W2 + j * MLP_H + k] * h1[k];
    out += fmaxf(z, 0.f) * th[P_W3 + j];
  }
  y[i] = out;
}

// ------------------------------------------------------------------ training

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// One minibatch's loss and gradient, fused: a CTA takes tiles of 32 samples
// through gather, forward and backward with the weights and the tile's
// activations in shared memory, keeps its share of the gradient in registers
// over its tiles and writes it once; k_reduce adds the CTAs' shares.  Every
// sum over inputs or units runs in the order of the plain loops (bias first,
// then index order), so the forward pass and the back-propagated values do
// not depend on the tiling; the sums over samples run per tile, then over the
// CTAs in a fixed order (deterministic, and shorter chains than one loop over
// the batch).
// What bounds it: a step is 127 MFLOP (B = 4096) spread over 128 CTAs, so the
// two launches' latency and the chain gather -> layers -> gradient, not a
// pipe.  The launches are chained (each becomes resident while the one before
// drains), and what another launch of the chain has written is read through
// L2.  Tiles of 32 give one CTA per SM at B = 4096; a thread's 2 x 4
// outputs of a layer take 6 16-byte shared loads per 32 FMAs.
// Measured on GB300, per step at B = 4096: 12 us (the ten separate kernels it
// replaces, one thread per output with strided global loads: 640 us).
constexpr int TT = 32;                 // samples per tile
constexpr int PART = 5316;             // floats per CTA in the partial buffer: 5313 parameters, loss, pad
constexpr int P_LOSS = MLP_PARAMS;
constexpr int SW1 = 20, SW2 = 68;      // shared row strides (floats): 16-byte rows on shifted banks

struct TrainSmem {
  alignas(16) float w1[MLP_H * SW1], w2[MLP_H * SW2];
  alignas(16) float x[TT * SW1];
  alignas(16) float h1[TT * SW2], h2[TT * SW2];  // activations, then in place dz1 and dz2
  float b1[MLP_H], b2[MLP_H], w3[MLP_H], b3;
  float t[TT], dy[TT], r2[TT];
};

// 2 samples x 4 units of act(W in + b): samples s0, s0 + 1, units u0 + 16 u.
template <int K>
__device__ __forceinline__ void layer_2x4(const float* in, int is, const float* W, int ws,
                                          const float* bias, int s0, int u0, float* out) {
  float z[2][4];
#pragma unroll
  for (int u = 0; u < 4; ++u) z[0][u] = z[1][u] = bias[u0 + 16 * u];
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    const float4 a = *reinterpret_cast<const float4*>(in + s0 * is + k);
    const float4 b = *reinterpret_cast<const float4*>(in + (s0 + 1) * is + k);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 w = *reinterpret_cast<const float4*>(W + (u0 + 16 * u) * ws + k);
      z[0][u] = fmaf(a.w, w.w, fmaf(a.z, w.z, fmaf(a.y, w.y, fmaf(a.x, w.x, z[0][u]))));
      z[1][u] = fmaf(b.w, w.w, fmaf(b.z, w.z, fmaf(b.y, w.y, fmaf(b.x, w.x, z[1][u]))));
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    out[s0 * SW2 + u0 + 16 * u] = fmaxf(z[0][u], 0.f);
    out[(s0 + 1) * SW2 + u0 + 16 * u] = fmaxf(z[1][u], 0.f);
  }
}

// idx: the batch's samples, or null to draw them by SplitMix64 on counter0 + b.
// stats: means and deviations that standardise X and T, or null for raw values.
__global__ void __launch_bounds__(256) k_minibatch(const float* __restrict__ th,
                                                   const float* __restrict__ X,
                                                   const float* __restrict__ T, int64_t n,
                                                   const int32_t* __restrict__ idx, uint64_t seed,
                                                   int64_t counter0, int B,
                                                   const float* __restrict__ stats,
                                                   float* __restrict__ part) {
  __shared__ TrainSmem sm;
  const int tid = threadIdx.x;
  // gather of a tile: 8 threads per sample, two features each; rows past the
  // batch take part with zeros and a zero output gradient.  The first tile's
  // samples do not depend on the step before, so their loads come ahead of
  // the wait for it; the next tile's go out before this one's arithmetic.
  float x0, x1, tv;
  auto gather = [&](int64_t b0) {
    const int s = tid >> 3, k = (tid & 7) * 2;
    const int64_t b = b0 + s;
    x0 = x1 = tv = 0.f;
    if (b < B) {
      const int64_t i = idx ? (int64_t)idx[b]
                            : (int64_t)(splitmix64(seed + (uint64_t)(counter0 + b)) % (uint64_t)n);
      x0 = X[i * MLP_IN + k];
      x1 = X[i * MLP_IN + k + 1];
      if (k == 0) tv = T[i];
      if (stats) {
        x0 = (x0 - stats[k]) / stats[MLP_IN + k];
        x1 = (x1 - stats[k + 1]) / stats[MLP_IN + k + 1];
        if (k == 0) tv = (tv - stats[2 * MLP_IN]) / stats[2 * MLP_IN + 1];
      }
    }
  };
  gather((int64_t)blockIdx.x * TT);
  chain();
  if (((uintptr_t)th & 15) == 0) {  // uniform
    const float4 v = __ldcg(reinterpret_cast<const float4*>(th + P_W1 + 4 * tid));
    float4 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = __ldcg(reinterpret_cast<const float4*>(th + P_W2 + 4 * (tid + 256 * q)));
    *reinterpret_cast<float4*>(sm.w1 + (tid >> 2) * SW1 + (tid & 3) * 4) = v;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = tid + 256 * q;
      *reinterpret_cast<float4*>(sm.w2 + (i >> 4) * SW2 + (i & 15) * 4) = w[q];
    }
  } else {
    for (int i = tid; i < MLP_H * MLP_IN; i += 256) sm.w1[(i >> 4) * SW1 + (i & 15)] = __ldcg(th + P_W1 + i);
    for (int i = tid; i < MLP_H * MLP_H; i += 256) sm.w2[(i >> 6) * SW2 + (i & 63)] = __ldcg(th + P_W2 + i);
  }
  if (tid < MLP_H) {
    sm.b1[tid] = __ldcg(th + P_B1 + tid);
    sm.b2[tid] = __ldcg(th + P_B2 + tid);
    sm.w3[tid] = __ldcg(th + P_W3 + tid);
  }
  if (tid == 0) sm.b3 = __ldcg(th + P_B3);
  const int tx = tid & 15, ty = tid >> 4;
  float g2[4][4], g1[4], gv = 0.f;  // W2, W1, and one of b2 / b1 / W3 / b3 / loss
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    g1[j] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) g2[j][i] = 0.f;
  }
  for (int64_t b0 = (int64_t)blockIdx.x * TT; b0 < B; b0 += (int64_t)gridDim.x * TT) {
    {
      const int s = tid >> 3, k = (tid & 7) * 2;
      sm.x[s * SW1 + k] = x0;
      sm.x[s * SW1 + k + 1] = x1;
      if (k == 0) sm.t[s] = tv;
    }
    gather(b0 + (int64_t)gridDim.x * TT);
    __syncthreads();
    layer_2x4<MLP_IN>(sm.x, SW1, sm.w1, SW1, sm.b1, 2 * ty, tx, sm.h1);
    __syncthreads();
    layer_2x4<MLP_H>(sm.h1, SW2, sm.w2, SW2, sm.b2, 2 * ty, tx, sm.h2);
    __syncthreads();
    if (tid < TT) {
      float y = sm.b3;
#pragma unroll 8
      for (int k = 0; k < MLP_H; k += 4) {
        const float4 h = *reinterpret_cast<const float4*>(sm.h2 + tid * SW2 + k);
        y = fmaf(h.w, sm.w3[k + 3], fmaf(h.z, sm.w3[k + 2], fmaf(h.y, sm.w3[k + 1], fmaf(h.x, sm.w3[k], y))));
      }
      const bool in = b0 + tid < B;
      const float r = in ? y - sm.t[tid] : 0.f;
      sm.dy[tid] = 2.f * r / (float)B;
      sm.r2[tid] = r * r;
    }
    __syncthreads();
    // gradients of W3, b3 and the loss; then h2 -> dz2 in place (each thread
    // its own elements; z2 > 0 exactly where h2 > 0)
    if (tid >= 128 && tid < 128 + MLP_H) {
      float s = 0.f;
      for (int b = 0; b < TT; ++b) s = fmaf(sm.dy[b], sm.h2[b * SW2 + tid - 128], s);
      gv += s;
    } else if (tid == 192 || tid == 193) {
      float s = 0.f;
      for (int b = 0; b < TT; ++b) s += tid == 192 ? sm.dy[b] : sm.r2[b];
      gv += s;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < TT * MLP_H / 256; ++k) {
      const int e = k * 256 + tid, b = e >> 6, j = e & 63;
      sm.h2[b * SW2 + j] = sm.h2[b * SW2 + j] > 0.f ? sm.dy[b] * sm.w3[j] : 0.f;
    }
    __syncthreads();
    // gW2[j][i] = sum_b dz2[b][j] h1[b][i], a 4 x 4 patch per thread
    {
      float p[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) p[j][i] = 0.f;
#pragma unroll 4
      for (int b = 0; b < TT; ++b) {
        const float4 d = *reinterpret_cast<const float4*>(sm.h2 + b * SW2 + 4 * ty);
        const float4 h = *reinterpret_cast<const float4*>(sm.h1 + b * SW2 + 4 * tx);
        const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) p[j][i] = fmaf(dv[j], hv[i], p[j][i]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) g2[j][i] += p[j][i];
    }
    if (tid < MLP_H) {
      float s = 0.f;
      for (int b = 0; b < TT; ++b) s += sm.h2[b * SW2 + tid];
      gv += s;
    }
    // dz1[b][i] = (sum_j dz2[b][j] W2[j][i]) (z1 > 0): 2 samples x 4 inputs
    float d1[2][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) d1[0][i] = d1[1][i] = 0.f;
#pragma unroll 4
    for (int j = 0; j < MLP_H; ++j) {
      const float4 w = *reinterpret_cast<const float4*>(sm.w2 + j * SW2 + 4 * tx);
      const float a = sm.h2[(2 * ty) * SW2 + j], b = sm.h2[(2 * ty + 1) * SW2 + j];
      d1[0][0] = fmaf(a, w.x, d1[0][0]);
      d1[0][1] = fmaf(a, w.y, d1[0][1]);
      d1[0][2] = fmaf(a, w.z, d1[0][2]);
      d1[0][3] = fmaf(a, w.w, d1[0][3]);
      d1[1][0] = fmaf(b, w.x, d1[1][0]);
      d1[1][1] = fmaf(b, w.y, d1[1][1]);
      d1[1][2] = fmaf(b, w.z, d1[1][2]);
      d1[1][3] = fmaf(b, w.w, d1[1][3]);
    }
    __syncthreads();  // every read of h1 is done
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float* h = sm.h1 + (2 * ty + q) * SW2 + 4 * tx + i;
        *h = *h > 0.f ? d1[q][i] : 0.f;
      }
    __syncthreads();
    // gW1[j][k] = sum_b dz1[b][j] x[b][k], four inputs per thread
    {
      const int j = tid >> 2, k = (tid & 3) * 4;
      float p[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int b = 0; b < TT; ++b) {
        const float d = sm.h1[b * SW2 + j];
        const float4 x = *reinterpret_cast<const float4*>(sm.x + b * SW1 + k);
        p[0] = fmaf(d, x.x, p[0]);
        p[1] = fmaf(d, x.y, p[1]);
        p[2] = fmaf(d, x.z, p[2]);
        p[3] = fmaf(d, x.w, p[3]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) g1[i] += p[i];
    }
    if (tid >= 64 && tid < 64 + MLP_H) {
      float s = 0.f;
      for (int b = 0; b < TT; ++b) s += sm.h1[b * SW2 + tid - 64];
      gv += s;
    }
    __syncthreads();  // the next tile overwrites x, h1 and h2
  }
  float* o = part + (int64_t)blockIdx.x * PART;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    *reinterpret_cast<float4*>(o + P_W2 + (4 * ty + j) * MLP_H + 4 * tx) =
        make_float4(g2[j][0], g2[j][1], g2[j][2], g2[j][3]);
  *reinterpret_cast<float4*>(o + P_W1 + 4 * tid) = make_float4(g1[0], g1[1], g1[2], g1[3]);
  if (tid < 64) o[P_B2 + tid] = gv;
  else if (tid < 128) o[P_B1 + tid - 64] = gv;
  else if (tid < 192) o[P_W3 + tid - 128] = gv;
  else if (tid == 192) o[P_B3] = gv;
  else if (tid == 193) o[P_LOSS] = gv;
}

// Sum of the G shares of 32 parameters per CTA (8 warps take every eighth
// share, then add up in order), followed by the Adam update (ADAM) or the
// store of the gradient.  Entry P_LOSS is the sum of squared residuals.
template <bool ADAM>
__global__ void __launch_bounds__(256) k_reduce(const float* __restrict__ part, int G, int B,
                                                float* __restrict__ grad, float* __restrict__ th,
                                                float* __restrict__ m, float* __restrict__ v,
                                                float lr, float c1, float c2,
                                                float* __restrict__ loss) {
  __shared__ float sh[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  float s = 0.f;
  chain();
  if (i <= P_LOSS) {
#pragma unroll 8
    for (int c = w; c < G; c += 8) s += __ldcg(part + (int64_t)c * PART + i);
  }
  sh[w][lane] = s;
  __syncthreads();
  if (w || i > P_LOSS) return;
  float g = sh[0][lane];
#pragma unroll
  for (int k = 1; k < 8; ++k) g += sh[k][lane];
  if (i == P_LOSS) {
    *loss = g / (float)B;
  } else if (ADAM) {
    const float mi = 0.9f * m[i] + 0.1f * g;
    const float vi = 0.999f * v[i] + 0.001f * g * g;
    m[i] = mi;
    v[i] = vi;
    th[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
  } else {
    grad[i] = g;
  }
}

// Column statistics (mean, standard deviation) of features and targets.
// A CTA takes rows of 64 (16 lanes per row, one column each, so X is read
// coalesced) and sums v - k and (v - k)^2 as pairs of floats, k = the column's
// first value: the variance does not cancel against a large mean, which the
// FP64 sums of v and v^2 did, on 17 CTAs.  Bound by DRAM (68 bytes per sample).
// The largest |v - k| goes along: k_stats_final sums a column again in FP64
// where squares have left FP32's range or k is far out.
constexpr int STAT_CTAS = 1216;  // eight per SM: the chains of dependent additions need the warps
constexpr int STAT_SUMS = 3 * (MLP_IN + 1);  // per CTA: sums of v - k and (v - k)^2, largest |v - k|
__global__ void __launch_bounds__(256) k_stats(const float* __restrict__ X,
                                               const float* __restrict__ T, int64_t n,
                                               double* __restrict__ part) {
  __shared__ double sh[2][16][17];
  __shared__ double st[2][256];
  __shared__ float mh[16][17], mt[256];
  const int c = threadIdx.x & 15, r = threadIdx.x >> 4;
  DD s1 = {0.f, 0.f}, s2 = {0.f, 0.f}, t1 = {0.f, 0.f}, t2 = {0.f, 0.f};
  float sm = 0.f, tm = 0.f;
  auto take = [](DD& a, DD& b, float& m, float v, float k) {
    const DD d = two_sum(v, -k);
    m = fmaxf(m, fabsf(d.h));
    dd_acc(a, d);
    const DD q = two_prod(d.h, d.h);
    dd_acc(b, {q.h, fmaf(2.f * d.h, d.l, q.l)});
  };
  const float kx = X[c], kt = T[0];
  for (int64_t i0 = (int64_t)blockIdx.x * 64; i0 < n; i0 += (int64_t)gridDim.x * 64) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t i = i0 + 16 * u + r;
      if (i < n) take(s1, s2, sm, X[i * MLP_IN + c], kx);
    }
    if (threadIdx.x < 64 && i0 + threadIdx.x < n) take(t1, t2, tm, T[i0 + threadIdx.x], kt);
  }
  sh[0][r][c] = (double)s1.h + s1.l;
  sh[1][r][c] = (double)s2.h + s2.l;
  st[0][threadIdx.x] = (double)t1.h + t1.l;
  st[1][threadIdx.x] = (double)t2.h + t2.l;
  mh[r][c] = sm;
  mt[threadIdx.x] = tm;
  __syncthreads();
  double* o = part + (int64_t)blockIdx.x * STAT_SUMS;
  if (threadIdx.x < 34) {
    const int k = threadIdx.x / 17, j = threadIdx.x - 17 * k;
    double a = 0.0;
    if (j < MLP_IN)
      for (int q = 0; q < 16; ++q) a += sh[k][q][j];
    else
      for (int q = 0; q < 64; ++q) a += st[k][q];
    o[threadIdx.x] = a;
  } else if (threadIdx.x >= 64 && threadIdx.x < 64 + 17) {
    const int j = threadIdx.x - 64;
    float m = 0.f;
    if (j < MLP_IN)
      for (int q = 0; q < 16; ++q) m = fmaxf(m, mh[q][j]);
    else
      for (int q = 0; q < 64; ++q) m = fmaxf(m, mt[q]);
    o[34 + j] = m;
  }
}

// Sums of a and b (and the largest m) over the CTA's 256 threads, in a fixed order,
// valid in thread 0.
__device__ __forceinline__ void stat_sums(double& a, double& b, float& m) {
  __shared__ double sa[8], sb[8];
  __shared__ float sm[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  }
  if ((threadIdx.x & 31) == 0) {
    sa[threadIdx.x >> 5] = a;
    sb[threadIdx.x >> 5] = b;
    sm[threadIdx.x >> 5] = m;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < 8; ++w) {
      a += sa[w];
      b += sb[w];
      m = fmaxf(m, sm[w]);
    }
}

// One CTA per column adds the CTAs' sums in a fixed order.  The pairs of floats
// are good to 2^-41 of each sum.  FP64 takes the column instead
//  - when a sum is not finite (|v - k| above 2^63, infinities, NaN);
//  - when the mean square of v - k is below 1e-30, where the low parts of the
//    squares leave FP32's range (but not for a constant column);
//  - when k is more than 32 deviations from the mean: b / n - d^2 would cancel
//    ten bits and more.
__global__ void __launch_bounds__(256) k_stats_final(const float* X, const float* T, int64_t n,
                                                    const double* __restrict__ part, int G,
                                                    float* stats) {
  const int c = blockIdx.x;  // 0..16 (16 = target)
  double a = 0.0, b = 0.0;
  float m = 0.f;
  for (int g = threadIdx.x; g < G; g += 256) {
    const double* p = part + (int64_t)g * STAT_SUMS + c;
    a += p[0];
    b += p[17];
    m = fmaxf(m, (float)p[34]);
  }
  stat_sums(a, b, m);
  __shared__ double mid;
  __shared__ bool again;
  double k = (double)(c < MLP_IN ? X[c] : T[0]);
  if (threadIdx.x == 0) {
    const double d = a / (double)n, ms = b / (double)n;
    again = !(isfinite(a) && isfinite(b)) || (m > 0.f && ms < 1e-30) || d * d > 1024.0 * (ms - d * d);
    mid = isfinite(k + d) ? k + d : 0.0;
  }
  __syncthreads();
  if (again) {
    k = mid;
    a = b = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += 256) {
      const double v = (double)(c < MLP_IN ? X[i * MLP_IN + c] : T[i]) - k;
      a += v;
      b += v * v;
    }
    stat_sums(a, b, m);
  }
  if (threadIdx.x == 0) {
    const double d = a / (double)n, mean = k + d;
    double var = b / (double)n - d * d;
    double sd = var > 0 ? sqrt(var) : 0.0;
    // constant column (the tau feature of a one-level set): a deviation below
    // 1e-6 of the mean's magnitude is rounding noise, and as a scale it would
    // blow up the folded first layer
    if (!(sd > 1e-30) || !(sd > 1e-6 * fabs(mean))) sd = 1.0;
    const int im = c < MLP_IN ? c : 2 * MLP_IN, is = c < MLP_IN ? MLP_IN + c : 2 * MLP_IN + 1;
    stats[im] = (float)mean;
    stats[is] = (float)sd;
  }
}

// Folds the normalisation into the first and last layers.
__global__ void __launch_bounds__(MLP_H) k_fold(float* th, const float* __restrict__ sv) {
  const int j = threadIdx.x;
  double b = th[P_B1 + j];
  for (int k = 0; k < MLP_IN; ++k) {
    const float w = th[P_W1 + j * MLP_IN + k];
    b -= (double)w * sv[k] / sv[MLP_IN + k];
    th[P_W1 + j * MLP_IN + k] = w / sv[MLP_IN + k];
  }
  th[P_B1 + j] = (float)b;
  th[P_W3 + j] *= sv[2 * MLP_IN + 1];
  if (j == 0) th[P_B3] = th[P_B3] * sv[2 * MLP_IN + 1] + sv[2 * MLP_IN];
}

// CTAs of a minibatch: one per tile of 32 samples, at most two per SM (a CTA
// then takes several tiles), which bounds the partial buffer to 6.5 MB.
static int minibatch_ctas(int B) {
  const int64_t tiles = ((int64_t)B + TT - 1) / TT;
  return (int)(tiles < 304 ? tiles : 304);
}
constexpr unsigned REDUCE_CTAS = (P_LOSS + 1 + 31) / 32;

struct DevBuf {
  void* p = nullptr;
  explicit DevBuf(size_t bytes) {
    if (bytes && cudaMalloc(&p, bytes) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
  }
  ~DevBuf() {
    if (p) cudaFree(p);
  }
  float* f() const { return (float*)p; }
};

// A training call's workspace (up to 7 MB), from a stream-ordered pool per device
// that keeps at most 64 MB between calls (pools grow by 32 MB; mapping them anew
// took 200 us of every call) and gives them back when a grid is destroyed.
static cudaMemPool_t work_pool(int device, bool create) {
  static std::mutex m;
  static cudaMemPool_t pools[64] = {};
  if (device < 0 || device >= 64) return nullptr;
  std::lock_guard<std::mutex> hold(m);
  if (!pools[device] && create) {
    cudaMemPoolProps p = {};
    p.allocType = cudaMemAllocationTypePinned;
    p.location.type = cudaMemLocationTypeDevice;
    p.location.id = device;
    uint64_t keep = 64ull << 20;
    if (cudaMemPoolCreate(&pools[device], &p) != cudaSuccess ||
        cudaMemPoolSetAttribute(pools[device], cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
      cudaGetLastError();
      pools[device] = nullptr;
    }
  }
  return pools[device];
}

void closure_trim(int device) {
  if (cudaMemPool_t p = work_pool(device, false)) cudaMemPoolTrimTo(p, 0);
}

struct StreamBuf {
  void* p = nullptr;
  cudaStream_t s;
  bool pooled = false;
  StreamBuf(size_t bytes, cudaStream_t st) : s(st) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaMemPool_t pool = work_pool(dev, true);
    pooled = pool && cudaMallocFromPoolAsync(&p, bytes, pool, s) == cudaSuccess;
    if (!pooled && cudaMalloc(&p, bytes) != cudaSuccess) p = nullptr;
    if (!pooled) cudaGetLastError();
  }
  ~StreamBuf() {
    if (p && pooled) cudaFreeAsync(p, s);
    else if (p) cudaFree(p);
  }
  float* f() const { return (float*)p; }
};

// ------------------------------------------------------------------- dataset

struct DsArgs {
  const void* f;  // fine populations (dense SoA)
  int nx, ny, nz, r, cx_, cy_, cz_;  // fine dims, filter, coarse dims
  int64_t N;
  float* sbar;   // 19 x nc shifted filtered populations
  float* mom;    // 10 x nc: rho, j (3), mean(j_a j_b / rho) (6: xx yy zz xy xz yz)
  float* num;    // nc
  float* den;    // nc
};

// The kernels below formed their sums, products and quotients in FP64 (some
// 230 operations per fine voxel and 350 per coarse one at two per SM and
// clock); as exact sums and pairs of floats (exact.cuh; results rounded to
// FP32, as before) they cost FP32 operations only.  Measured on GB300, 256^3
// FP32, r = 2, one dataset call: 8.5 ms -> 0.55 ms.

// Coordinates of the calling thread's coarse voxel; false past the end.
__device__ __forceinline__ bool cvoxel(const DsArgs& a, int64_t& X, int& x, int& y, int& z) {
  X = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (X >= (int64_t)a.cx_ * a.cy_ * a.cz_) return false;
  const int row = (int)(X / a.cx_);
  x = (int)(X - (int64_t)row * a.cx_);
  z = row / a.cy_;
  y = row - z * a.cy_;
  return true;
}

// One coarse voxel's filter in FP64.
template <int S> __device__ __noinline__ void filter_f64(const DsArgs& a, int64_t X, int Xx, int Xy, int Xz) {
  using T = typename Codec<S>::T;
  const int64_t nc = (int64_t)a.cx_ * a.cy_ * a.cz_;
  double sp[Q], m[10];
  for (int i = 0; i < Q; ++i) sp[i] = 0;
  for (int k = 0; k < 10; ++k) m[k] = 0;
  for (int dz = 0; dz < a.r; ++dz)
    for (int dy = 0; dy < a.r; ++dy) {
      const T* f = (const T*)a.f + (Xx * a.r + (int64_t)a.nx * ((Xy * a.r + dy) + (int64_t)a.ny * (Xz * a.r + dz)));
      for (int dx = 0; dx < a.r; ++dx, ++f) {
        double rho = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          const double fi = Codec<S>::abs_d(f[(int64_t)i * a.N], i);
          sp[i] += fi - wd(i);
          rho += fi;
          jx += cx(i) * fi;
          jy += cy(i) * fi;
          jz += cz(i) * fi;
        }
        m[0] += rho;
        m[1] += jx;
        m[2] += jy;
        m[3] += jz;
        m[4] += jx * jx / rho;
        m[5] += jy * jy / rho;
        m[6] += jz * jz / rho;
        m[7] += jx * jy / rho;
        m[8] += jx * jz / rho;
        m[9] += jy * jz / rho;
      }
    }
  const double inv = 1.0 / ((double)a.r * a.r * a.r);
  for (int i = 0; i < Q; ++i) a.sbar[(int64_t)i * nc + X] = (float)(sp[i] * inv);
  for (int k = 0; k < 10; ++k) a.mom[(int64_t)k * nc + X] = (float)(m[k] * inv);
}

// mean of n values whose sum is s, minus w, to FP32.  pow2: n is a power of two
// (uniform), so n w and the scaling are exact.
__device__ __forceinline__ float mean_minus(DD s, float n, bool pow2, DD inv_n, float wh, float wl) {
  if (pow2) {
    const DD t = two_sum(s.h, -(n * wh)), x = two_sum(t.h, s.l);
    return add_rn(x.h, add_rn(x.l, sub_rn(t.l, n * wl))) * inv_n.h;
  }
  s = two_sum(s.h, s.l);
  const DD q = two_prod(n, wh), d = two_sum(s.h, -q.h);
  const DD t = quick_sum(d.h, add_rn(d.l, sub_rn(s.l, fmaf(n, wl, q.l))));
  return dd_mul(t, inv_n).h;
}

// rho and j of a fine voxel outside the exact sums' window, from FP64.  False if
// pairs of floats cannot go on with them (infinities, NaN, magnitudes that
// products or quotients would carry out of FP32's range).
__device__ __noinline__ bool filter_wide(const float v[Q], bool shifted, DD* out) {
  double m = 0, x = 0, y = 0, z = 0;
  bool in = true;
  for (int i = 0; i < Q; ++i) {
    in = in && fabsf(v[i]) < 0x1p30f;
    const double f = shifted ? wd(i) + (double)v[i] : (double)v[i];
    m += f;
    x += cx(i) * f;
    y += cy(i) * f;
    z += cz(i) * f;
  }
  const double d[4] = {m, x, y, z};
  for (int k = 0; k < 4; ++k) {
    out[k].h = (float)d[k];
    out[k].l = (float)(d[k] - (double)out[k].h);
  }
  return in && fabs(m) > 0x1p-30;
}

// One thread per coarse voxel.  rho and j of each fine voxel are exact.  The sums
// over the fine voxels:
//   r <= 3, FP32 and FP16: the population sums add the split parts without
//     rounding (per voxel an upper part counts at most 2^15 (FP32) or 2^19 (FP16)
//     units, a lower one 2^19, and 2^19 r^3 <= 2^24).  A coarse voxel with a
//     value outside the window takes the FP64 form as a whole;
//   PAIRS, r <= 16: pairs of floats, renormalised after each row, so that their
//     error stays below r^4 2^-48 of the sum of magnitudes (2^-32); any
//     magnitude will do, and voxels outside the window take rho and j from
//     FP64.  BF16 takes this form at r <= 3 too: its values reach below the
//     window wherever s crosses zero.
// Wider filters are left to the FP64 form.  One dataset call at 256^3, r = 2,
// FP32 and FP16: 0.55 ms with the split parts, 0.67 with pairs; r = 4: 0.45
// (FP64: 6.9 and 7.5).
template <int S, bool PAIRS>
__global__ void __launch_bounds__(128) k_ds_filter(const __grid_constant__ DsArgs a) {
  using T = typename Codec<S>::T;
  const int64_t nc = (int64_t)a.cx_ * a.cy_ * a.cz_;
  int64_t X;
  int Xx, Xy, Xz;
  if (!cvoxel(a, X, Xx, Xy, Xz)) return;
  DD sp[Q], m[10];
#pragma unroll
  for (int i = 0; i < Q; ++i) sp[i] = {0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 10; ++k) m[k] = {0.f, 0.f};
  bool in = true;
#pragma unroll 1
  for (int dz = 0; dz < a.r; ++dz)
#pragma unroll 1
    for (int dy = 0; dy < a.r; ++dy) {
      const T* f = (const T*)a.f + (Xx * a.r + (int64_t)a.nx * ((Xy * a.r + dy) + (int64_t)a.ny * (Xz * a.r + dz)));
#pragma unroll 1
      for (int dx = 0; dx < a.r; ++dx, ++f) {
        float v[Q];
        static_for<Q>([&](auto ic) {
          constexpr int i = decltype(ic)::value;
          if constexpr (S == S_F32) v[i] = f[(int64_t)i * a.N];
          else v[i] = Codec<S>::template load<i>(f[(int64_t)i * a.N]);
        });
        FixSum<S> q;
        DD c[4];
        {
          float h[Q], l[Q];
          const bool ok = FixSum<S>::split(v, h, l);
          if (!q.pairs(h, l, ok, c)) in = PAIRS && filter_wide(v, S != S_F32, c) && in;
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            if constexpr (PAIRS) {
              dd_acc(sp[i], v[i]);
            } else {
              sp[i].h = add_rn(sp[i].h, h[i]);
              sp[i].l = add_rn(sp[i].l, l[i]);
            }
          }
        }
        const DD inv = dd_inv(c[0]);
        const DD ux = dd_mul(c[1], inv), uy = dd_mul(c[2], inv), uz = dd_mul(c[3], inv);
#pragma unroll
        for (int k = 0; k < 4; ++k) dd_acc(m[k], c[k]);
        dd_acc(m[4], dd_prod(c[1], ux));
        dd_acc(m[5], dd_prod(c[2], uy));
        dd_acc(m[6], dd_prod(c[3], uz));
        dd_acc(m[7], dd_prod(c[1], uy));
        dd_acc(m[8], dd_prod(c[1], uz));
        dd_acc(m[9], dd_prod(c[2], uz));
      }
      if constexpr (PAIRS) {
#pragma unroll
        for (int i = 0; i < Q; ++i) sp[i] = two_sum(sp[i].h, sp[i].l);
#pragma unroll
        for (int k = 0; k < 10; ++k) m[k] = two_sum(m[k].h, m[k].l);
      }
    }
  if (!in) {
    filter_f64<S>(a, X, Xx, Xy, Xz);
    return;
  }
  const float n = (float)(a.r * a.r * a.r);
  const DD inv = dd_inv({n, 0.f});
  const bool pow2 = (a.r & (a.r - 1)) == 0;
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    constexpr float wh = S == S_F32 ? (float)wd(i) : 0.f;
    constexpr float wl = S == S_F32 ? (float)(wd(i) - (double)(float)wd(i)) : 0.f;
    a.sbar[(int64_t)i * nc + X] = mean_minus(sp[i], n, pow2, inv, wh, wl);
  });
#pragma unroll
  for (int k = 0; k < 10; ++k) a.mom[(int64_t)k * nc + X] = mean_minus(m[k], n, pow2, inv, 0.f, 0.f);
}

template <int S> __global__ void __launch_bounds__(128) k_ds_filter_f64(const __grid_constant__ DsArgs a) {
  int64_t X;
  int x, y, z;
  if (cvoxel(a, X, x, y, z)) filter_f64<S>(a, X, x, y, z);
}

template <int S> static void ds_filter(const DsArgs& a, unsigned nb, cudaStream_t s) {
  if (a.r <= 3 && S != S_BF16) k_ds_filter<S, false><<<nb, 128, 0, s>>>(a);
  else if (a.r <= 16) k_ds_filter<S, true><<<nb, 128, 0, s>>>(a);
  else k_ds_filter_f64<S><<<nb, 128, 0, s>>>(a);
}

// Index of a coarse voxel with every coordinate in [-1, c].
__device__ __forceinline__ int64_t cidx(const DsArgs& a, int x, int y, int z) {
  auto wrap = [](int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); };
  return wrap(x, a.cx_) + (int64_t)a.cx_ * (wrap(y, a.cy_) + (int64_t)a.cy_ * wrap(z, a.cz_));
}

__global__ void __launch_bounds__(128) k_ds_features(DsArgs a, float tau, float* feats) {
  const int64_t nc = (int64_t)a.cx_ * a.cy_ * a.cz_;
  int64_t X;
  int x, y, z;
  if (!cvoxel(a, X, x, y, z)) return;
  float s[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) s[i] = a.sbar[(int64_t)i * nc + cidx(a, x - cx(i), y - cy(i), z - cz(i))];
  float xf[MLP_IN];
  closure_features(s, tau, xf);
  float* o = feats + X * MLP_IN;
  if (((uintptr_t)feats & 15) == 0) {  // uniform: the rows are 64 bytes
#pragma unroll
    for (int k = 0; k < MLP_IN; k += 4)
      *reinterpret_cast<float4*>(o + k) = make_float4(xf[k], xf[k + 1], xf[k + 2], xf[k + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) o[k] = xf[k];
  }
}

// Numerator and denominator of the least-squares eddy viscosity.
__global__ void __launch_bounds__(128) k_ds_numden(DsArgs a) {
  const int64_t nc = (int64_t)a.cx_ * a.cy_ * a.cz_;
  int64_t X;
  int x, y, z;
  if (!cvoxel(a, X, x, y, z)) return;
  // j / rho of FP32 values: quotient and remainder
  auto vel = [&](int64_t i, DD u[3]) {
    const float r = a.mom[i], w = 1.f / r;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float j = a.mom[(int64_t)(1 + b) * nc + i], q = mul_rn(j, w);
      u[b] = quick_sum(q, mul_rn(fmaf(-q, r, j), w));
    }
  };
  DD g[3][3];  // g[a][b] = 2 d u_b / d x_a
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    DD p[3], m[3];
    vel(cidx(a, x + (d == 0), y + (d == 1), z + (d == 2)), p);
    vel(cidx(a, x - (d == 0), y - (d == 1), z - (d == 2)), m);
#pragma unroll
    for (int b = 0; b < 3; ++b) g[d][b] = dd_add(p[b], neg(m[b]));
  }
  DD u[3];
  vel(X, u);
  // sub-filter stress: mean(j_a j_b / rho) - j_a u_b
  DD t[6];  // xx yy zz xy xz yz
  auto stress = [&](int k, int p, int q) {
    const float j = a.mom[(int64_t)(1 + p) * nc + X];
    const DD e = two_prod(j, u[q].h);
    t[k] = dd_add({a.mom[(int64_t)(4 + k) * nc + X], 0.f}, neg(quick_sum(e.h, fmaf(j, u[q].l, e.l))));
  };
  stress(0, 0, 0);
  stress(1, 1, 1);
  stress(2, 2, 2);
  stress(3, 0, 1);
  stress(4, 0, 2);
  stress(5, 1, 2);
  const DD third = {0x1.555556p-2f, -0x1.555556p-27f};
  const DD tr = dd_mul(dd_add(dd_add(t[0], t[1]), t[2]), third);
  DD num = {0.f, 0.f}, den = {0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 3; ++i) {  // S_ii = g_ii / 2
    const DD s = {0.5f * g[i][i].h, 0.5f * g[i][i].l};
    num = dd_add(num, dd_mul(dd_add(t[i], neg(tr)), s));
    den = dd_add(den, dd_mul(s, s));
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {  // 2 S_ij = (g_ij + g_ji) / 2, twice in the sums
    const int i = k == 2 ? 1 : 0, j = k == 0 ? 1 : 2;
    const DD e = dd_add(g[i][j], g[j][i]);
    const DD s2 = {0.5f * e.h, 0.5f * e.l};
    num = dd_add(num, dd_mul(t[3 + k], s2));
    const DD q = dd_mul(s2, s2);
    den = dd_add(den, {0.5f * q.h, 0.5f * q.l});
  }
  a.num[X] = num.h;
  a.den[X] = dd_mul(den, {2.f * a.mom[X], 0.f}).h;
}

__global__ void __launch_bounds__(128) k_ds_target(DsArgs a, float tau, float* targets) {
  int64_t X;
  int x, y, z;
  if (!cvoxel(a, X, x, y, z)) return;
  DD n = {0.f, 0.f}, d = {0.f, 0.f};
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        const int64_t i = cidx(a, x + dx, y + dy, z + dz);
        dd_acc(n, a.num[i]);
        dd_acc(d, a.den[i]);
      }
  n = two_sum(n.h, n.l);  // n may cancel
  d = quick_sum(d.h, d.l);
  float t = 0.f;
  if (d.h > 1e-30f) {
    const DD q = dd_mul(n, dd_inv(d)), p = two_prod(-3.f, q.h);
    t = add_rn(p.h, fmaf(-3.f, q.l, p.l));
  } else if (d.h > 0.f) {  // 1 / d would overflow
    t = (float)(-3.0 * ((double)n.h + n.l) / ((double)d.h + d.l));
  }
  const float lo = (float)(-((double)tau - 0.5) + 1e-3);
  t = t < lo ? lo : (t > 0.5f ? 0.5f : t);
  targets[X] = t;
}

}  // namespace lbm

using namespace lbm;

extern "C" {

lbm_status lbm_closure_forward(const float* theta, const float* feats, int64_t n, int bf16,
                               float* out, void* stream) {
  set_error("");
  if (!theta || !feats || !out || n <= 0) return fail(LBM_ERR_INVALID, "bad closure_forward arguments");
  cudaStream_t s = (cudaStream_t)stream;
  if (!bf16) {
    k_mlp_forward_fp32<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(theta, feats, n, out);
    LBM_CUDA(cudaGetLastError());
    return LBM_OK;
  }
  // BF16 copy of the weights (device), as lbm_closure_load builds it
  std::vector<float> h(MLP_PARAMS);
  LBM_CUDA(cudaMemcpyAsync(h.data(), theta, MLP_PARAMS * sizeof(float), cudaMemcpyDeviceToHost, s));
  LBM_CUDA(cudaStreamSynchronize(s));
  ClosureParams cp;
  closure_params_from_fp32(h.data(), &cp);
  DevBuf d(sizeof(ClosureParams));
  if (!d.p) return fail(LBM_ERR_OOM, "device allocation failed");
  LBM_CUDA(cudaMemcpyAsync(d.p, &cp, sizeof(cp), cudaMemcpyHostToDevice, s));
  k_mlp_forward_bf16<<<(unsigned)((n + 255) / 256), 256, 0, s>>>((const ClosureParams*)d.p, feats, n, out);
  LBM_CUDA(cudaGetLastError());
  LBM_CUDA(cudaStreamSynchronize(s));
  return LBM_OK;
}

lbm_status lbm_closure_grad(const float* theta, const float* feats, const float* targets,
                            const int32_t* idx, int batch, float* grad, float* loss, void* stream) {
  set_error("");
  if (!theta || !feats || !targets || !idx || !grad || !loss || batch <= 0)
    return fail(LBM_ERR_INVALID, "bad closure_grad arguments");
  cudaStream_t s = (cudaStream_t)stream;
  const int G = minibatch_ctas(batch);
  DevBuf part((size_t)G * PART * sizeof(float));
  if (!part.p) return fail(LBM_ERR_OOM, "device allocation failed");
  k_minibatch<<<G, 256, 0, s>>>(theta, feats, targets, 0, idx, 0, 0, batch, nullptr, part.f());
  k_reduce<false><<<REDUCE_CTAS, 256, 0, s>>>(part.f(), G, batch, grad, nullptr, nullptr, nullptr, 0.f, 1.f,
                                              1.f, loss);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? LBM_OK : cuda_fail(e, "closure_grad");
}

lbm_status lbm_closure_train(const float* feats, const float* targets, int64_t n, int steps,
                             int batch, float lr, uint64_t seed, float* theta_io, float* loss_out,
                             void* stream) {
  set_error("");
  if (!feats || !targets || !theta_io || n <= 0 || steps <= 0 || batch <= 0)
    return fail(LBM_ERR_INVALID, "bad closure_train arguments");
  cudaStream_t s = (cudaStream_t)stream;
  // one allocation: the CTAs' gradient shares, Adam's moments, the last loss
  // and the column statistics
  const int G = minibatch_ctas(batch);
  const size_t n_part = (size_t)G * PART;
  StreamBuf buf((n_part + 2 * PART + 64) * sizeof(float) + STAT_CTAS * STAT_SUMS * sizeof(double), s);
  lbm_status st = buf.p ? LBM_OK : fail(LBM_ERR_OOM, "device allocation failed");
  if (!st) {
    float *part = buf.f(), *m = part + n_part, *v = m + PART, *stats = v + PART, *loss = stats + 48;
    double* spart = reinterpret_cast<double*>(stats + 64);  // an even number of floats from the base
    const int SG = (int)(n < STAT_CTAS * 64LL ? (n + 63) / 64 : STAT_CTAS);
    cudaMemsetAsync(m, 0, 2 * PART * sizeof(float), s);
    k_stats<<<SG, 256, 0, s>>>(feats, targets, n, spart);
    k_stats_final<<<MLP_IN + 1, 256, 0, s>>>(feats, targets, n, spart, SG, stats);
    for (int it = 1; it <= steps; ++it) {
      launch_step(it > 1, k_minibatch, G, 256, 0, s, theta_io, feats, targets, n, nullptr, seed,
                  (int64_t)(it - 1) * batch, batch, stats, part);
      const float c1 = 1.f - powf(0.9f, (float)it), c2 = 1.f - powf(0.999f, (float)it);
      launch_step(true, k_reduce<true>, REDUCE_CTAS, 256, 0, s, part, G, batch, nullptr, theta_io, m, v, lr, c1,
                  c2, loss);
    }
    k_fold<<<1, MLP_H, 0, s>>>(theta_io, stats);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && loss_out)
      e = cudaMemcpyAsync(loss_out, loss, sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) st = cuda_fail(e, "closure_train");
  }
  return st;
}

lbm_status lbm_closure_dataset(lbm_grid* h, int r, double tau_coarse, float* feats,
                               float* targets) {
  set_error("");
  if (!h || !feats || !targets || r < 1) return fail(LBM_ERR_INVALID, "bad closure_dataset arguments");
  Grid& g = h->g;
  if (g.kind != 0 || g.q != 19)
    return fail(LBM_ERR_UNSUPPORTED, "closure datasets come from dense D3Q19 grids");
  Level& L = g.lv[0];
  for (int a = 0; a < 3; ++a)
    if (!g.phys.periodic[a]) return fail(LBM_ERR_UNSUPPORTED, "closure datasets need a periodic box");
  if (L.nx % r || L.ny % r || L.nz % r) return fail(LBM_ERR_INVALID, "dims must be multiples of r");
  lbm_status st = lbm_sync(h);
  if (st) return st;
  DsArgs a{};
  a.f = L.f[L.cur];
  a.nx = L.nx;
  a.ny = L.ny;
  a.nz = L.nz;
  a.r = r;
  a.cx_ = L.nx / r;
  a.cy_ = L.ny / r;
  a.cz_ = L.nz / r;
  a.N = L.n_slots;
  const int64_t nc = (int64_t)a.cx_ * a.cy_ * a.cz_;
  // Workspace: 31 floats per coarse voxel (260 MB at 256^3, r = 2), kept with the
  // grid up to 512 MB (550 us a call; 819 with an allocation in each).
  // (The buffer that the next step overwrites would do for its size, but walls
  // set later leave solid voxels whose stored values the caller can read.)
  const size_t need = (size_t)nc * (Q + 12) * 4;
  constexpr size_t kWorkKeep = (size_t)512 << 20;
  std::lock_guard<std::mutex> hold(g.work_mutex);
  if (need <= kWorkKeep && need > g.work_bytes) {
    g.dfree(g.work_d, g.stream);
    g.work_d = g.dalloc(need, g.stream);
    g.work_bytes = g.work_d ? need : 0;
  }
  const bool kept = need <= g.work_bytes;
  DevBuf own(kept ? 0 : need);
  if (!kept && !own.p) return fail(LBM_ERR_OOM, "device allocation failed");
  a.sbar = kept ? (float*)g.work_d : own.f();
  a.mom = a.sbar + nc * Q;
  a.num = a.mom + nc * 10;
  a.den = a.num + nc;
  cudaStream_t s = g.stream;
  const unsigned nb = (unsigned)((nc + 127) / 128);
  switch (g.phys.storage) {
    case S_F32: ds_filter<S_F32>(a, nb, s); break;
    case S_F16: ds_filter<S_F16>(a, nb, s); break;
    default: ds_filter<S_BF16>(a, nb, s); break;
  }
  k_ds_features<<<nb, 128, 0, s>>>(a, (float)tau_coarse, feats);
  k_ds_numden<<<nb, 128, 0, s>>>(a);
  k_ds_target<<<nb, 128, 0, s>>>(a, (float)tau_coarse, targets);
  LBM_CUDA(cudaGetLastError());
  LBM_CUDA(cudaStreamSynchronize(s));
  return LBM_OK;
}

lbm_status lbm_closure_load(lbm_grid* h, const float* theta, size_t n) {
  set_error("");
  if (!h || !theta) return fail(LBM_ERR_INVALID, "NULL argument");
  if (n != (size_t)MLP_PARAMS) return fail(LBM_ERR_INVALID, "closure weights must have 5313 values");
  Grid& g = h->g;
  if (g.kind != 2 || g.q != 19)
    return fail(LBM_ERR_UNSUPPORTED, "the closure runs on D3Q19 multi-resolution grids");
  ClosureParams cp;
  closure_params_from_fp32(theta, &cp);
  if (!g.closure_d) {
    g.closure_d = g.dalloc(sizeof(ClosureParams), g.stream);
    if (!g.closure_d) return fail(LBM_ERR_OOM, "device allocation failed");
  }
  LBM_CUDA(cudaMemcpyAsync(g.closure_d, &cp, sizeof(cp), cudaMemcpyHostToDevice, g.stream));
  LBM_CUDA(cudaStreamSynchronize(g.stream));
  g.closure_loaded = true;
  return LBM_OK;
}

}  // extern "C"
