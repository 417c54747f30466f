// fields.cu - layout-generic kernels: FP64 equilibrium initialisation,
// moments, FP64 population decode and the conservation reduction.
//
// A voxel (x, y, z) of a level's virtual box maps to storage as
//   dense : index(pop) = pop * N + v,                 v = x + nx (y + ny z)
//   sparse: index(pop) = (b * Q + pop) * E^3 + l,     b = block id from the
//           virtual block map, l = lx + E (ly + E lz)
#include "d3q19.cuh"
#include "exact.cuh"
#include "grid.h"

namespace lbm {
namespace LBM_LNS {

struct LevelDev {
  int nx, ny, nz, E, nbx, nby, nbz;
  int64_t N;  // dense: voxels; sparse: slots
  const uint8_t* flags;  // dense: per voxel (may be null); sparse: per slot
  const int32_t* bmap;
};

static LevelDev level_dev(const Level& L) {
  LevelDev d;
  d.nx = L.nx;
  d.ny = L.ny;
  d.nz = L.nz;
  d.E = L.E;
  d.nbx = L.nbx;
  d.nby = L.nby;
  d.nbz = L.nbz;
  d.N = L.n_slots;
  d.flags = L.flags_d;
  d.bmap = L.bmap_d;
  return d;
}

// Storage base / stride of the virtual-box voxel with linear id v; false if
// no storage exists.  DENSE needs no coordinates.
template <bool DENSE>
__device__ __forceinline__ bool locate(const LevelDev& d, int64_t v, int64_t& base,
                                       int64_t& stride, uint8_t& flag) {
  if constexpr (DENSE) {
    base = v;
    stride = d.N;
    flag = d.flags ? d.flags[v] : (uint8_t)0;
    return true;
  }
  int x, y, z;
  if (v <= 0xffffffffLL) {
    const uint32_t w = (uint32_t)v, row = w / (uint32_t)d.nx;
    x = (int)(w - row * (uint32_t)d.nx);
    z = (int)(row / (uint32_t)d.ny);
    y = (int)(row - (uint32_t)z * (uint32_t)d.ny);
  } else {
    const int64_t row = v / d.nx;
    x = (int)(v - row * d.nx);
    z = (int)(row / d.ny);
    y = (int)(row - (int64_t)z * d.ny);
  }
  const int e = d.E == 8 ? 3 : 2, M = d.E - 1;
  const int b = d.bmap[(x >> e) + d.nbx * ((y >> e) + d.nby * (z >> e))];
  if (b < 0) return false;
  const int l = (x & M) + (((y & M) + ((z & M) << e)) << e);
  stride = (int64_t)1 << (3 * e);
  base = (int64_t)b * Q * stride + l;
  flag = d.flags[(int64_t)b * stride + l];
  return true;
}

// FP64 forms, for values outside the windows of the exact ones.
template <int S>
__device__ __noinline__ void init_wide(typename Codec<S>::T* out, int64_t stride, double r, double ux,
                                       double uy, double uz) {
#pragma unroll
  for (int i = 0; i < Q; ++i) out[i * stride] = Codec<S>::from_double(feq_d(i, r, ux, uy, uz), i);
}

template <int S>
__device__ __noinline__ void sums_wide(const typename Codec<S>::T* in, int64_t stride, double r[4]) {
  double m = 0, x = 0, y = 0, z = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const double fi = Codec<S>::abs_d(in[i * stride], i);
    m += fi;
    if (cx(i)) x += cx(i) * fi;
    if (cy(i)) y += cy(i) * fi;
    if (cz(i)) z += cz(i) * fi;
  }
  r[0] = m;
  r[1] = x;
  r[2] = y;
  r[3] = z;
}

// Stored values as floats (FP32: f, 16-bit: s = f - w).
template <int S>
__device__ __forceinline__ void load_raw(const typename Codec<S>::T* in, int64_t stride, float v[Q]) {
  static_for<Q>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    if constexpr (S == S_F32) v[i] = in[i * stride];
    else v[i] = Codec<S>::template load<i>(in[i * stride]);
  });
}

// Initial state, moments and conservation sums.  In FP64 they were bound by
// that pipe (29 us per operation and voxel at 256^3: some 190, 125 and 68 of
// them); with the exact sums and pairs of floats they move DRAM traffic.
// Measured on GB300, 256^3 FP32, init + moments + conservation: 10.49 ms ->
// 1.05 ms (DRAM floor 0.73 ms).
template <int S, bool DENSE>
__global__ void __launch_bounds__(256, 6) k_init_eq(LevelDev d, void* f, const double* __restrict__ rho,
                                                 const double* __restrict__ u) {
  using T = typename Codec<S>::T;
  const int64_t n = (int64_t)d.nx * d.ny * d.nz;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    int64_t base, stride;
    uint8_t fl;
    if (!locate<DENSE>(d, v, base, stride, fl)) continue;
    if (!type_updated(flag_type(fl))) continue;
    const double r = rho ? rho[v] : 1.0;
    const double ux = u ? u[v] : 0.0, uy = u ? u[n + v] : 0.0, uz = u ? u[2 * n + v] : 0.0;
    T* out = (T*)f + base;
    EqPair q;
    bool sure = q.set(r, ux, uy, uz);
    if (sure)
      q.all([&](auto ic, DD e) {
        constexpr int i = decltype(ic)::value;
        out[i * stride] = eq_store<S>(i, e, sure);
      });
    if (!sure) init_wide<S>(out, stride, r, ux, uy, uz);
  }
}

// Six CTAs per SM (40 registers) against the five that 48 allow: 256^3, D3Q19
// FP32 402 -> 369 us, FP16 380 -> 369, D3Q27 FP32 495 -> 429, but D3Q27 FP16
// 412 -> 443, which is left to the compiler.
template <int S, bool DENSE>
__global__ void __launch_bounds__(256, Q == 27 && S != S_F32 ? 0 : 6)
    k_moments(LevelDev d, const void* f, double* __restrict__ rho, double* __restrict__ u) {
  using T = typename Codec<S>::T;
  const int64_t n = (int64_t)d.nx * d.ny * d.nz;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    int64_t base, stride;
    uint8_t fl;
    double r = nan, ux = nan, uy = nan, uz = nan;
    if (locate<DENSE>(d, v, base, stride, fl) && type_updated(flag_type(fl))) {
      const T* in = (const T*)f + base;
      float g[Q];
      load_raw<S>(in, stride, g);
      FixSum<S> q;
      if (q.set(g)) {
        fix_moments<S>(q, r, ux, uy, uz);
      } else {
        double w[4];
        sums_wide<S>(in, stride, w);
        r = w[0];
        ux = w[1] / r;
        uy = w[2] / r;
        uz = w[3] / r;
      }
    }
    if (rho) rho[v] = r;
    if (u) {
      u[v] = ux;
      u[n + v] = uy;
      u[2 * n + v] = uz;
    }
  }
}

template <int S, bool DENSE>
__global__ void k_decode(LevelDev d, const void* f, double* dst) {
  using T = typename Codec<S>::T;
  const int64_t n = (int64_t)d.nx * d.ny * d.nz;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    int64_t base, stride;
    uint8_t fl;
    const bool ok = locate<DENSE>(d, v, base, stride, fl) && type_updated(flag_type(fl));
    const T* in = (const T*)f;
#pragma unroll
    for (int i = 0; i < Q; ++i)
      dst[i * n + v] = ok ? Codec<S>::abs_d(in[base + i * stride], i) : nan;
  }
}

// ---------------------------------------------------------------- reduction
// Pass 1: every CTA reduces a fixed, grid-strided set of slots to 4 doubles
// (per thread an exact 64-bit fixed-point sum and, for voxels outside its
// window, an FP64 one; then warp shuffles and shared memory) and writes them
// to partials[cta].  A thread adds at most N / 233,472 voxels below 2^46
// units each: no overflow.
// Pass 2: one CTA adds the partials in a fixed order.  The result does not
// depend on scheduling, so repeated calls give bit-identical sums.
constexpr int RED_THREADS = 256;
// Six CTAs per SM, all resident: 258 us at 256^3 FP32 (307 with 1216 CTAs, four
// resident per SM).
constexpr int RED_CTAS = 912;
static_assert(RED_CTAS <= kRedCtas, "partials of one level");

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <int S>
__global__ void __launch_bounds__(RED_THREADS, 6) k_cons_partial(LevelDev d, const void* f,
                                                              double weight, double* partials) {
  using T = typename Codec<S>::T;
  const T* in = (const T*)f;
  double acc[4] = {0, 0, 0, 0};
  int64_t fix[4] = {0, 0, 0, 0};
  const int e = d.E == 0 ? 0 : (d.E == 8 ? 9 : 6);  // log2 of a block's voxels
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < d.N;
       s += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t fl = d.flags ? d.flags[s] : (uint8_t)0;
    if (!type_updated(flag_type(fl))) continue;
    const int64_t stride = e == 0 ? d.N : (int64_t)1 << e;
    const T* p = in + (e == 0 ? s : (s >> e) * Q * stride + (s & (stride - 1)));
    float g[Q];
    load_raw<S>(p, stride, g);
    FixSum<S> q;
    if (q.set(g)) {
      fix[0] += q.m;
      fix[1] += q.x;
      fix[2] += q.y;
      fix[3] += q.z;
    } else {
      double w[4];
      sums_wide<S>(p, stride, w);
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[k] += w[k];
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) acc[k] += (double)fix[k] * (1.0 / (double)FixSum<S>::ONE);
  __shared__ double sh[RED_THREADS / 32][4];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double w = warp_sum(acc[k]);
    if (lane == 0) sh[wid][k] = w;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0;
    for (int w = 0; w < RED_THREADS / 32; ++w) t += sh[w][threadIdx.x];
    partials[blockIdx.x * 4 + threadIdx.x] = t * weight;
  }
}

__global__ void __launch_bounds__(RED_THREADS) k_cons_final(const double* partials, int n,
                                                            double* out4) {
  double acc[4] = {0, 0, 0, 0};
  for (int p = threadIdx.x; p < n; p += blockDim.x)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] += partials[p * 4 + k];
  __shared__ double sh[RED_THREADS / 32][4];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double w = warp_sum(acc[k]);
    if (lane == 0) sh[wid][k] = w;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0;
    for (int w = 0; w < RED_THREADS / 32; ++w) t += sh[w][threadIdx.x];
    out4[threadIdx.x] = t;
  }
}

// ------------------------------------------------------------------ launchers
static unsigned grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > 152 * 64) b = 152 * 64;
  if (b < 1) b = 1;
  return (unsigned)b;
}

template <int S>
static void launch_k_init_eq(const LevelDev& d, unsigned nb, cudaStream_t s, void* f, const double* rho,
                             const double* u) {
  if (d.E == 0) k_init_eq<S, true><<<nb, 256, 0, s>>>(d, f, rho, u);
  else k_init_eq<S, false><<<nb, 256, 0, s>>>(d, f, rho, u);
}
template <int S>
static void launch_k_moments(const LevelDev& d, unsigned nb, cudaStream_t s, const void* f, double* rho,
                             double* u) {
  if (d.E == 0) k_moments<S, true><<<nb, 256, 0, s>>>(d, f, rho, u);
  else k_moments<S, false><<<nb, 256, 0, s>>>(d, f, rho, u);
}
template <int S>
static void launch_k_decode(const LevelDev& d, unsigned nb, cudaStream_t s, const void* f, double* dst) {
  if (d.E == 0) k_decode<S, true><<<nb, 256, 0, s>>>(d, f, dst);
  else k_decode<S, false><<<nb, 256, 0, s>>>(d, f, dst);
}

lbm_status launch_init_equilibrium(Grid& g, Level& L, const double* rho, const double* u,
                                   cudaStream_t s) {
  const LevelDev d = level_dev(L);
  const int64_t n = (int64_t)L.nx * L.ny * L.nz;
  const unsigned nb = grid_for(n, 256);
  switch (g.phys.storage) {
    case S_F32: launch_k_init_eq<S_F32>(d, nb, s, L.f[L.cur], rho, u); break;
    case S_F16: launch_k_init_eq<S_F16>(d, nb, s, L.f[L.cur], rho, u); break;
    default: launch_k_init_eq<S_BF16>(d, nb, s, L.f[L.cur], rho, u); break;
  }
  LBM_CUDA(cudaGetLastError());
  return LBM_OK;
}

lbm_status launch_moments(Grid& g, Level& L, double* rho, double* u, cudaStream_t s) {
  const LevelDev d = level_dev(L);
  const int64_t n = (int64_t)L.nx * L.ny * L.nz;
  const unsigned nb = grid_for(n, 256);
  switch (g.phys.storage) {
    case S_F32: launch_k_moments<S_F32>(d, nb, s, L.f[L.cur], rho, u); break;
    case S_F16: launch_k_moments<S_F16>(d, nb, s, L.f[L.cur], rho, u); break;
    default: launch_k_moments<S_BF16>(d, nb, s, L.f[L.cur], rho, u); break;
  }
  LBM_CUDA(cudaGetLastError());
  return LBM_OK;
}

lbm_status launch_decode_f64(Grid& g, Level& L, double* dst, cudaStream_t s) {
  const LevelDev d = level_dev(L);
  const int64_t n = (int64_t)L.nx * L.ny * L.nz;
  const unsigned nb = grid_for(n, 256);
  switch (g.phys.storage) {
    case S_F32: launch_k_decode<S_F32>(d, nb, s, L.f[L.cur], dst); break;
    case S_F16: launch_k_decode<S_F16>(d, nb, s, L.f[L.cur], dst); break;
    default: launch_k_decode<S_BF16>(d, nb, s, L.f[L.cur], dst); break;
  }
  LBM_CUDA(cudaGetLastError());
  return LBM_OK;
}

lbm_status launch_conservation(Grid& g, double* out4, cudaStream_t s) {
  int np = 0;
  for (int l = 0; l < g.n_levels; ++l) {
    Level& L = g.lv[l];
    const LevelDev d = level_dev(L);
    unsigned nb = (unsigned)((L.n_slots + RED_THREADS - 1) / RED_THREADS);
    if (nb > (unsigned)RED_CTAS) nb = RED_CTAS;
    if (nb < 1) nb = 1;
    const double w = (double)(1LL << (3 * l));  // 8^l volume weight
    double* part = g.partials_d + (size_t)np * 4;
    switch (g.phys.storage) {
      case S_F32: k_cons_partial<S_F32><<<nb, RED_THREADS, 0, s>>>(d, L.f[L.cur], w, part); break;
      case S_F16: k_cons_partial<S_F16><<<nb, RED_THREADS, 0, s>>>(d, L.f[L.cur], w, part); break;
      default: k_cons_partial<S_BF16><<<nb, RED_THREADS, 0, s>>>(d, L.f[L.cur], w, part); break;
    }
    np += (int)nb;
  }
  k_cons_final<<<1, RED_THREADS, 0, s>>>(g.partials_d, np, out4);
  LBM_CUDA(cudaGetLastError());
  return LBM_OK;
}

}  // namespace LBM_LNS
}  // namespace lbm
