// Host build of csrc/exact.cuh (test_exact_host.py): every form against plain
// FP64, integer or long double arithmetic, over seeded states of its whole window.
// Prints "name value" lines.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
// device-only calls of d3q19.cuh, not reached here
inline void cudaGridDependencySynchronize() {}
inline void cudaTriggerProgrammaticLaunchCompletion() {}
#include "exact.cuh"

using namespace lbm;
using Long = long double;

static std::mt19937_64 gen(20260);
static double uniform(double a, double b) { return a + (b - a) * (double)(gen() >> 11) * 0x1p-53; }
static double sign() { return gen() & 1 ? -1.0 : 1.0; }

template <int S> static float stored(double v) {
  if constexpr (S == S_F32) return (float)v;
  if constexpr (S == S_F16) return __half2float(__float2half_rn((float)v));
  return __bfloat162float(__float2bfloat16_rn((float)v));
}

// One value of kind k: around equilibrium, over the whole window, at random
// exponents, equal lower parts, zeros.
template <int S> static float value(int k, int i) {
  const double top = S == S_F32 ? 1.9999 : 0.4995, bot = S == S_F32 ? 0x1p-11 : -top;
  double v;
  switch (k % 6) {
    case 0: v = wd(i) * (S == S_F32 ? uniform(0.7, 1.3) : uniform(-0.3, 0.3)); break;
    case 1: v = uniform(bot, top); break;
    case 2: v = std::ldexp(uniform(1, 2), -(int)(gen() % (S == S_F32 ? 11 : 30)) - (S == S_F32 ? 0 : 2)) *
                (S == S_F32 ? 1.0 : sign()); break;
    case 3: v = (S == S_F32 ? wd(i) : -0.04) + 0.49 * (S == S_F32 ? 0x1p-14 : 0x1p-20); break;
    case 4: v = S == S_F32 ? wd(i) * 0.07 + 0x1p-11 : -0.9 * wd(i) + 0.4 * 0x1p-20; break;
    default: v = (S == S_F32 || gen() % 3) ? (S == S_F32 ? wd(i) * uniform(1, 20) : uniform(-0.05, 0.05)) : 0.0;
  }
  v = v > top ? top : v;
  return stored<S>(S == S_F32 && v < bot ? bot : v);
}

template <int S> static void moments(const char* name) {
  long sums = 0, quotients = 0, rejected = 0, taken = 0;
  for (int k = 0; k < 600000; ++k) {
    float v[Q];
    int64_t m = S == S_F32 ? 0 : FixSum<S>::ONE, x = 0, y = 0, z = 0;
    for (int i = 0; i < Q; ++i) {
      v[i] = value<S>(k, i);
      const int64_t f = (int64_t)std::ldexp((double)v[i], FixSum<S>::FRAC);
      m += f;
      x += cx(i) * f;
      y += cy(i) * f;
      z += cz(i) * f;
    }
    FixSum<S> q;
    if (!q.set(v)) {
      ++rejected;
      continue;
    }
    ++taken;
    sums += q.m != m || q.x != x || q.y != y || q.z != z;
    double r, ux, uy, uz;
    fix_moments<S>(q, r, ux, uy, uz);
    // both operands are exact doubles, so the host's quotient is the rounded one
    const double w = (double)m;
    quotients += r != std::ldexp(w, -FixSum<S>::FRAC) || ux != (double)x / w || uy != (double)y / w || uz != (double)z / w;
  }
  std::printf("%s_wrong_sums %ld\n%s_wrong_quotients %ld\n%s_taken %ld\n%s_rejected %ld\n", name, sums, name, quotients,
              name, taken, name, rejected);
}

static void quotients() {
  long wrong = 0;
  for (int k = 0; k < 4000000; ++k) {
    int64_t m = (int64_t)(gen() >> (17 + gen() % 17)), x = (int64_t)(gen() >> (17 + gen() % 46));
    if (m == 0) m = 1;
    if (k % 16 == 0) x = m << (gen() % 3);                       // a power of two
    if (k % 16 == 1) x = m - 1 - (int64_t)(gen() % 3);           // just below one
    if (k % 16 == 2) x = m + 1 + (int64_t)(gen() % 3);
    if (x >= (int64_t)1 << 47) x >>= 3;
    if (gen() & 1) x = -x;
    const double want = (double)x / (double)m;
    uint64_t b;
    std::memcpy(&b, &want, 8);
    for (int d = -1; d <= 1 && x; ++d) {  // starting values one unit off either way
      double q = bits_d(b + (uint64_t)(int64_t)d);
      wrong += round_quotient(x, m, q) != want;
    }
    if (x == 0) wrong += round_quotient(0, m, 0.0) != 0.0;
  }
  std::printf("wrong_round_quotient %ld\n", wrong);
}

static void equilibrium() {
  Long worst = 0;
  long rejected = 0, unsure[3] = {0, 0, 0}, differ[3] = {0, 0, 0};
  for (int k = 0; k < 400000; ++k) {
    double rho = uniform(0.9, 1.1), u[3];
    for (double& v : u) v = uniform(-0.249, 0.249) * (k & 3 ? 0.3 : 1.0);
    if (k % 7 == 0) u[k % 3] = 0.0;
    if (k % 11 == 0) u[k % 3] = sign() * std::ldexp(uniform(1, 2), -(int)(gen() % 58) - 3);
    if (k % 13 == 0) rho = std::ldexp(uniform(1, 2), (int)(gen() % 16) - 8);
    EqPair q;
    if (!q.set(rho, u[0], u[1], u[2])) {
      ++rejected;
      continue;
    }
    q.all([&](auto ic, DD f) {
      constexpr int i = decltype(ic)::value;
      const Long c = cx(i) * (Long)u[0] + cy(i) * (Long)u[1] + cz(i) * (Long)u[2];
      const Long s = (Long)u[0] * u[0] + (Long)u[1] * u[1] + (Long)u[2] * u[2];
      const Long want = (Long)wd(i) * rho * (1 + 3 * c + 4.5L * c * c - 1.5L * s);
      const Long e = std::fabs(((Long)f.h + (Long)f.l - want) / want);
      worst = e > worst ? e : worst;
    });
  }
  std::printf("equilibrium_log2_error %.3f\nequilibrium_rejected %ld\n", (double)std::log2(worst), rejected);
}

int main() {
  moments<S_F32>("f32");
  moments<S_F16>("f16");
  moments<S_BF16>("bf16");
  quotients();
  equilibrium();
  // windows
  DD r;
  const double refused[] = {0.25, -0.3, 0x1p-61, 1e-300, INFINITY, NAN};
  int taken = 0;
  for (double v : refused) taken += split<-60, -2>(v, r);
  std::printf("split_taken_outside %d\n", taken);
  float v[Q];
  int outside = 0;
  for (float bad : {INFINITY, -INFINITY, NAN, 2.f, -0.1f, 0x1p-12f}) {
    for (int i = 0; i < Q; ++i) v[i] = wf(i);
    v[3] = bad;
    FixSum<S_F32> q;
    outside += q.set(v);
  }
  for (float bad : {INFINITY, -INFINITY, NAN, 0.5f, -0.75f}) {
    for (int i = 0; i < Q; ++i) v[i] = 0.f;
    v[3] = bad;
    FixSum<S_F16> q;
    FixSum<S_BF16> p;
    outside += q.set(v) + p.set(v);
  }
  for (int i = 0; i < Q; ++i) v[i] = 0.f;
  v[2] = 0x1p-34f;
  FixSum<S_BF16> p;
  outside += p.set(v);
  std::printf("sums_taken_outside %d\n", outside);
  return 0;
}
