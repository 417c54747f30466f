// exact.cuh - sums and products beyond FP32 without the FP64 pipe (internal).
//
// GB300 issues two FP64 operations per SM and clock against 128 FP32 ones, so
// a kernel that does FP64 arithmetic per population is bound by that pipe
// long before DRAM.  Two replacements live here:
//  - sums of stored populations as exact integers: each value is split into
//    two FP32 parts on fixed grids, the parts are added without rounding
//    (every partial sum is a multiple of the grid unit below 2^24 of them),
//    and the two sums form one 64-bit fixed-point number;
//  - pairs of floats (value h + l, |l| <= ulp(h) / 2: Dekker, Numer. Math. 18,
//    1971; Knuth, TAOCP vol. 2, 4.2.2) where products and quotients are
//    needed: about 46 bits, enough for results that are rounded to FP32.
// Values outside the stated windows (and infinities and NaN) are left to FP64
// code by the caller.
#pragma once
#include <cstring>

#include "d3q19.cuh"

namespace lbm {

// Single roundings, never contracted into other operations.
__host__ __device__ __forceinline__ float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
__host__ __device__ __forceinline__ float sub_rn(float a, float b) { return add_rn(a, -b); }
__host__ __device__ __forceinline__ float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ __forceinline__ uint32_t f_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t u;
  memcpy(&u, &f, 4);
  return u;
#endif
}
__host__ __device__ __forceinline__ float bits_f(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  memcpy(&f, &u, 4);
  return f;
#endif
}
__host__ __device__ __forceinline__ uint64_t d_bits(double d) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(d);
#else
  uint64_t u;
  memcpy(&u, &d, 8);
  return u;
#endif
}
__host__ __device__ __forceinline__ double bits_d(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double d;
  memcpy(&d, &u, 8);
  return d;
#endif
}

// ------------------------------------------------------------ pairs of floats

struct DD {
  float h, l;
};

// a + b, |a| >= |b| (or a's exponent not below b's).
__host__ __device__ __forceinline__ DD quick_sum(float a, float b) {
  const float s = add_rn(a, b);
  return {s, sub_rn(b, sub_rn(s, a))};
}
// a + b in any order.
__host__ __device__ __forceinline__ DD two_sum(float a, float b) {
  const float s = add_rn(a, b), t = sub_rn(s, a);
  return {s, add_rn(sub_rn(a, sub_rn(s, t)), sub_rn(b, t))};
}
__host__ __device__ __forceinline__ DD two_prod(float a, float b) {
  const float p = mul_rn(a, b);
  return {p, fmaf(a, b, -p)};
}
__host__ __device__ __forceinline__ DD neg(DD a) { return {-a.h, -a.l}; }
__host__ __device__ __forceinline__ DD dd_add(DD a, DD b) {
  const DD s = two_sum(a.h, b.h);
  return quick_sum(s.h, add_rn(s.l, add_rn(a.l, b.l)));
}
// The same without renormalising: l may exceed half an ulp of h.
__host__ __device__ __forceinline__ DD dd_sum(DD a, DD b) {
  const DD s = two_sum(a.h, b.h);
  return {s.h, add_rn(s.l, add_rn(a.l, b.l))};
}
__host__ __device__ __forceinline__ DD dd_mul(DD a, DD b) {
  const DD p = two_prod(a.h, b.h);
  return quick_sum(p.h, fmaf(a.h, b.l, fmaf(a.l, b.h, p.l)));
}
// dd_mul without renormalising, for sums.
__host__ __device__ __forceinline__ DD dd_prod(DD a, DD b) {
  const DD p = two_prod(a.h, b.h);
  return {p.h, fmaf(a.h, b.l, fmaf(a.l, b.h, p.l))};
}
// Accumulate x (or a pair) without renormalising: s.l collects the errors.
__host__ __device__ __forceinline__ void dd_acc(DD& s, float x) {
  const DD t = two_sum(s.h, x);
  s.h = t.h;
  s.l = add_rn(s.l, t.l);
}
__host__ __device__ __forceinline__ void dd_acc(DD& s, DD x) {
  const DD t = two_sum(s.h, x.h);
  s.h = t.h;
  s.l = add_rn(s.l, add_rn(t.l, x.l));
}
// 1 / a for a normal a.h.
__host__ __device__ __forceinline__ DD dd_inv(DD a) {
  const float r = 1.f / a.h;
  const float e = fmaf(-a.l, r, fmaf(-a.h, r, 1.f));
  return quick_sum(r, mul_rn(r, e));
}

// Split of a double: h its leading 24 bits (truncated), l the other 29
// rounded to 24.  False (h, l unspecified) unless a is 0 or 2^LO <= |a| <
// 2^HI, with LO >= -60 and HI <= 100.
template <int LO, int HI>
__host__ __device__ __forceinline__ bool split(double a, DD& r) {
  const uint64_t u = d_bits(a);
  const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
  const uint32_t e = (hi >> 20) & 0x7ffu;
  const bool zero = ((hi << 1) | lo) == 0u;
  // the low eight bits of the exponent, rebased by 896 = 1023 - 127
  const uint32_t m = (((uint32_t)(u >> 29) & 0x7fffffffu) ^ 0x40000000u) | (hi & 0x80000000u);
  const float l = (float)(int32_t)(lo & 0x1fffffffu) * bits_f((e - 948u) << 23);
  r.h = zero ? 0.f : bits_f(m);
  r.l = zero ? 0.f : bits_f(f_bits(l) ^ (hi & 0x80000000u));
  return zero || e - (uint32_t)(1023 + LO) < (uint32_t)(HI - LO);
}

namespace LBM_LNS {

// ------------------------------------------------------- exact moment sums
// rho and j of one voxel as 64-bit fixed-point numbers.
//   FP32 storage    every f in [2^-11, 2): the upper part is the nearest
//                   multiple of 2^-14, the lower one (|.| <= 2^-15) a multiple
//                   of 2^-34, the last bit of the smallest f.  Sums of 27:
//                   below 54 / 2^-14 < 2^20 and 27 2^-15 / 2^-34 < 2^24 units.
//   16-bit storage  every s = f - w zero or 2^-33 <= |s| < 1/2: upper unit
//                   2^-20, lower part (|.| <= 2^-21) a multiple of 2^-40 (BF16
//                   has eight bits; FP16 ends at 2^-24).  Sums of 27 below
//                   14 / 2^-20 < 2^24 and 27 2^-21 / 2^-40 < 2^24 units.
// In both the lower sum counts 2^-20 of the upper unit.
template <int S> struct FixSum {
  static constexpr int FRAC = S == S_F32 ? 34 : 40;  // fraction bits
  static constexpr int64_t ONE = (int64_t)1 << FRAC;
  int64_t m, x, y, z;  // rho, j
  float rho;           // rho in FP32 (a starting value for its reciprocal)

  // v: the stored values as floats (FP32: f; 16-bit: s).  False if a value
  // is outside the window or rho is not in [1/16, 64).  parts: the sums of
  // the upper and lower parts (rho, j; without the 1 of 16-bit storage).
  __host__ __device__ __forceinline__ bool set(const float v[Q]) {
    float a[4], b[4];
    const bool ok = parts(v, a, b);
    m = fix(a[0], b[0]) + (S == S_F32 ? 0 : ONE);
    x = fix(a[1], b[1]);
    y = fix(a[2], b[2]);
    z = fix(a[3], b[3]);
    return ok;
  }
  __host__ __device__ __forceinline__ bool parts(const float v[Q], float a[4], float b[4]) {
    float h[Q], l[Q];
    const bool ok = split(v, h, l);
    sums(h, a);
    sums(l, b);
    rho = total(a[0], b[0]);
    return ok && rho >= 0.0625f && rho < 64.f;
  }
  // The two parts of each value (v = h + l always); whether all are in the window.
  __host__ __device__ static __forceinline__ bool split(const float v[Q], float h[Q], float l[Q]) {
    constexpr float UP = S == S_F32 ? 768.f : 12.f;  // 1.5 2^23 upper units
    constexpr uint32_t LOW = (S == S_F32 ? 127u - 11u : 127u - 33u) << 23;
    constexpr uint32_t TOP = (S == S_F32 ? 128u : 126u) << 23;
    uint32_t mn = 0xffffffffu, mx = 0u;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if constexpr (S == S_F32) {
        const uint32_t u = f_bits(v[i]);
        mn = u < mn ? u : mn;
        mx = u > mx ? u : mx;
      } else {
        const uint32_t u = f_bits(v[i]) & 0x7fffffffu;
        if constexpr (S == S_BF16) mn = u - 1u < mn ? u - 1u : mn;  // zero wraps to the largest
        mx = u > mx ? u : mx;
      }
      h[i] = sub_rn(add_rn(v[i], UP), UP);
      l[i] = sub_rn(v[i], h[i]);
    }
    bool ok = mx < TOP;
    if constexpr (S == S_F32) ok = ok && mn >= LOW;
    if constexpr (S == S_BF16) ok = ok && mn >= LOW - 1u;
    return ok;
  }
  // From split parts: rho, j as pairs of floats.
  __host__ __device__ __forceinline__ bool pairs(const float h[Q], const float l[Q], bool ok, DD c[4]) {
    float a[4], b[4];
    sums(h, a);
    sums(l, b);
    rho = total(a[0], b[0]);
    c[0] = two_sum(a[0], b[0]);
    if (S != S_F32) {
      const DD s = two_sum(1.f, c[0].h);
      c[0] = quick_sum(s.h, add_rn(s.l, c[0].l));
    }
#pragma unroll
    for (int k = 1; k < 4; ++k) c[k] = two_sum(a[k], b[k]);
    return ok && rho >= 0.0625f && rho < 64.f;
  }

 private:
  // rho to FP32 (1 + a is exact): the reciprocal's third-order step needs all 24 bits
  __host__ __device__ static __forceinline__ float total(float a, float b) {
    return S == S_F32 ? add_rn(a, b) : add_rn(add_rn(1.f, a), b);
  }
  __host__ __device__ static __forceinline__ void sums(const float p[Q], float r[4]) {
    float m = p[0], x = 0.f, y = 0.f, z = 0.f;
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const float d = sub_rn(p[i], p[i + 1]);
      m = add_rn(m, add_rn(p[i], p[i + 1]));
      if (cx(i)) x = add_rn(x, cx(i) > 0 ? d : -d);
      if (cy(i)) y = add_rn(y, cy(i) > 0 ? d : -d);
      if (cz(i)) z = add_rn(z, cz(i) > 0 ? d : -d);
    }
    r[0] = m;
    r[1] = x;
    r[2] = y;
    r[3] = z;
  }
  __host__ __device__ static __forceinline__ int to_int(float v) {
#ifdef __CUDA_ARCH__
    return __float2int_rn(v);
#else
    return (int)v;
#endif
  }
  __host__ __device__ static __forceinline__ int64_t fix(float h, float l) {
    constexpr float A = (float)((int64_t)1 << (FRAC - 20)), B = (float)ONE;
    return ((int64_t)to_int(h * A) << 20) + (int64_t)to_int(l * B);
  }
};

// x / m rounded to nearest, from a double q within two units in its last place:
// the remainder |x| 2^-e - Q m of q = Q 2^e is a small integer, so 64-bit products
// and shifts modulo 2^64 give it exactly, and the remainder over m says by how many
// units q is off.  |x|, m < 2^47, q < 2^52 (no ties: a quotient of such numbers has
// no 54-bit form).  Next to a power of two, where the unit changes, the quotient
// is formed anew.  (A correction by two FP64 operations per quotient would cost
// 170 us at 256^3; the integer one costs 7 to 30.)
__host__ __device__ __forceinline__ double round_quotient(int64_t x, int64_t m, double q) {
  constexpr uint64_t FRACTION = ((uint64_t)1 << 52) - 1;
  const uint64_t b = d_bits(q), low = b & FRACTION;
  const int shift = 1075 - (int)((b >> 52) & 0x7ffu);  // -e
  const uint64_t a = (uint64_t)(x < 0 ? -x : x);
  const int64_t r = (int64_t)((shift < 64 ? a << shift : 0) - (low + FRACTION + 1) * (uint64_t)m);
  if (x == 0 || r == 0) return q;
  if (((low + 2) & FRACTION) < 4) return (double)x / (double)m;
  const int64_t r2 = 2 * r, m3 = 3 * m;
  return bits_d(b + (uint64_t)((r2 > m) + (r2 > m3) - (r2 < -m) - (r2 < -m3)));
}

// rho and u = j / rho as doubles: rho is exact; 1 / rho comes from the FP32
// reciprocal by one third-order step (relative error below 2^-52.9), u is one
// product, then rounded to nearest.  Ten FP64 operations; scalings by powers of two
// and the conversion of the FP32 value go through the exponent bits.
template <int S>
__host__ __device__ __forceinline__ void fix_moments(const FixSum<S>& f, double& r, double& ux, double& uy,
                                                     double& uz) {
  // |sums| < 2^47: exact as the low mantissa bits of 1.5 2^52
  auto dbl = [](int64_t v) { return bits_d((uint64_t)(0x4338000000000000LL + v)) - 6755399441055744.0; };
  const double m = dbl(f.m);  // rho 2^FRAC, positive
  r = bits_d(d_bits(m) - ((uint64_t)FixSum<S>::FRAC << 52));
#ifdef __CUDA_ARCH__
  const uint32_t b = f_bits(__frcp_rn(f.rho));  // in (1/64, 16]: normal
#else
  const uint32_t b = f_bits(1.f / f.rho);
#endif
  double y = bits_d(((uint64_t)((b >> 3) + (uint32_t)((896 - FixSum<S>::FRAC) << 20)) << 32) | (uint64_t)(b << 29));
  const double e = fma(-m, y, 1.0);
  y = fma(y, fma(e, e, e), y);
  ux = round_quotient(f.x, f.m, dbl(f.x) * y);
  uy = round_quotient(f.y, f.m, dbl(f.y) * y);
  uz = round_quotient(f.z, f.m, dbl(f.z) * y);
}

// ------------------------------------------------------------- equilibrium
// f^eq_i from double inputs in pairs of floats, before the last rounding: the
// even part h = 1 + c^2 / 2 - 3/2 u.u and the odd part c = 3 c_i.u of a pair of
// opposite directions are shared.  out(i, p) receives f^eq_i as a pair with
// a relative error below 2^-42.5.  Needs 2^-8 <= rho < 2^8 and |u_a| < 1/4 (0 or
// >= 2^-60): then |h| > |c|.
struct EqPair {
  DD rho, u[3];
  __host__ __device__ __forceinline__ bool set(double r, double x, double y, double z) {
    const bool a = split<-8, 8>(r, rho) && rho.h > 0.f;
    const bool b = split<-60, -2>(x, u[0]), c = split<-60, -2>(y, u[1]), d = split<-60, -2>(z, u[2]);
    return a && b && c && d;
  }
  template <class OUT> __host__ __device__ __forceinline__ void all(OUT&& out) const {
    DD v[3], R[4];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const DD p = two_prod(3.f, u[a].h);
      v[a] = quick_sum(p.h, fmaf(3.f, u[a].l, p.l));
    }
    // 1 - 3/2 u.u
    DD s = dd_add(dd_add(dd_mul(v[0], u[0]), dd_mul(v[1], u[1])), dd_mul(v[2], u[2]));
    const DD b = dd_add({1.f, 0.f}, {-0.5f * s.h, -0.5f * s.l});
    constexpr int first[4] = {0, 1, 7, Q - 1};
#pragma unroll
    for (int k = 0; k < (Q == 27 ? 4 : 3); ++k) {
      const float wh = (float)wd(first[k]), wl = (float)(wd(first[k]) - (double)(float)wd(first[k]));
      R[k] = dd_mul(DD{wh, wl}, rho);
    }
    out(IC<0>{}, scaled(R[0], b));
    static_for<(Q - 1) / 2>([&](auto pc) {
      constexpr int i = 2 * decltype(pc)::value + 1;
      constexpr int cls = i < 7 ? 1 : (i < 19 ? 2 : 3);
      DD c = {0.f, 0.f};
      bool have = false;
      auto take = [&](int e, DD q) {
        if (e == 0) return;
        const DD t = e > 0 ? q : neg(q);
        c = have ? dd_sum(c, t) : t;
        have = true;
      };
      take(cx(i), v[0]);
      take(cy(i), v[1]);
      take(cz(i), v[2]);
      // c^2 / 2
      const float hc = 0.5f * c.h;
      const float p = mul_rn(hc, c.h), pl = fmaf(c.h, c.l, fmaf(hc, c.h, -p));
      const DD h = two_sum(b.h, p);
      const float hl = add_rn(h.l, add_rn(b.l, pl));
      const DD f = quick_sum(h.h, c.h), g = quick_sum(h.h, -c.h);
      out(IC<i>{}, scaled(R[cls], {f.h, add_rn(f.l, add_rn(hl, c.l))}));
      out(IC<i + 1>{}, scaled(R[cls], {g.h, add_rn(g.l, sub_rn(hl, c.l))}));
    });
  }

 private:
  __host__ __device__ static __forceinline__ DD scaled(DD R, DD t) {
    const float p = mul_rn(R.h, t.h);
    return {p, fmaf(R.h, t.l, fmaf(R.l, t.h, fmaf(R.h, t.h, -p)))};
  }
};

// A pair as a float that rounds like it: FP32 storage takes the nearest, 16-bit
// storage h + l - w rounded to odd, so that the second rounding is that of the
// exact sum.
template <int S> __host__ __device__ __forceinline__ float eq_value(int i, DD f) {
  if constexpr (S == S_F32) {
    return add_rn(f.h, f.l);
  } else {
    const float wh = (float)wd(i), wl = (float)(wd(i) - (double)(float)wd(i));
    const DD d = two_sum(f.h, -wh);
    const DD s = two_sum(d.h, add_rn(d.l, sub_rn(f.l, wl)));
    const uint32_t u = f_bits(s.h);
    // away from zero: the error has the sum's sign
    const bool even = !(u & 1u) && s.l != 0.f && s.h != 0.f;
    const bool out = ((f_bits(s.l) ^ u) >> 31) == 0u;
    return bits_f(even ? (out ? u + 1u : u - 1u) : u);
  }
}

// The stored value of f^eq_i, and whether every value within 2^-42 of the pair
// rounds to it; where not (two voxels in ten thousand, FP32) the caller
// evaluates in FP64, so the state is the one that FP64 gives.
template <int S>
__host__ __device__ __forceinline__ typename Codec<S>::T eq_store(int i, DD f, bool& sure) {
  const float e = fabsf(f.h) * 0x1p-42f;
  const float a = eq_value<S>(i, {f.h, sub_rn(f.l, e)}), b = eq_value<S>(i, {f.h, add_rn(f.l, e)});
  if constexpr (S == S_F32) {
    sure = sure && a == b;
    return a;
  } else {
    typename Codec<S>::T s, t;
    if constexpr (S == S_F16) {
      s = __float2half_rn(a);
      t = __float2half_rn(b);
      sure = sure && __half2float(s) == __half2float(t);
    } else {
      s = __float2bfloat16_rn(a);
      t = __float2bfloat16_rn(b);
      sure = sure && __bfloat162float(s) == __bfloat162float(t);
    }
    return s;
  }
}

}  // namespace LBM_LNS
}  // namespace lbm
