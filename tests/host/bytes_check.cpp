// Host check of the byte slicing (csrc/qs_bytes.cuh): digits, packed words,
// exact levels with started accumulators, recombination against 128-bit
// integers, and whole dot products against exact sums.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "qs_bytes.cuh"

using namespace qsby;
typedef __int128 i128;

static uint32_t hi(double x) { uint64_t u; memcpy(&u, &x, 8); return (uint32_t)(u >> 32); }
static uint32_t lo(double x) { uint64_t u; memcpy(&u, &x, 8); return (uint32_t)u; }
static int fail(const char* what) { printf("FAIL %s\n", what); return 1; }

static std::mt19937_64 rng(7);
static double draw(int spread) {
  std::uniform_real_distribution<double> u(1.0, 2.0);
  double x = u(rng);
  if (rng() % 8 == 0) x = 2.0 - std::ldexp((double)(1 + rng() % 3), -52);        // all ones
  if (rng() % 16 == 0) x = 2.0 - std::ldexp(1.0, -(int)(5 + rng() % 5));          // around the row_field bump
  if (rng() % 16 == 0) x = 1.0;
  if (rng() % 16 == 0) return rng() % 2 ? 0.0 : -0.0;
  return std::ldexp(x, -(int)(rng() % (uint64_t)(spread + 1))) * (rng() % 2 ? 1.0 : -1.0);
}

// digits, rounding, packing of one row
static int check_row(int spread, int base) {
  double x[8];
  uint32_t mx = 0;
  for (double& v : x) {
    v = std::ldexp(draw(spread), base);
    const uint32_t m = hi(v) & 0x7FFFFFFFu;
    if (m > mx) mx = m;
  }
  const uint32_t ef = row_field(mx);
  const int E = (int)(ef >> 20) - 1023;
  uint64_t T[8];
  for (int i = 0; i < 8; ++i) {
    T[i] = bytes_of(hi(x[i]), lo(x[i]), ef + 0x100000u);
    i128 V = 0;
    for (int s = 0; s < kA; ++s) {
      const int d = digit_a(T[i], s);
      if (d < -128 || d > 127) return fail("digit range");
      V = V * 256 + d;
    }
    const long double want = std::ldexp((long double)x[i], 54 - E);
    if (std::fabs((double)((long double)V - want)) > 0.5 + 1.0 / 256) return fail("digit value");
  }
  for (int i = 0; i < 8; i += 2) {
    uint32_t w[7];
    packed_digits(T[i], T[i + 1], w);
    for (int s = 0; s < kA; ++s)
      if ((int)(w[s] & 0xFFFFu) != digit_a(T[i], s) + 128 || (int)(w[s] >> 16) != digit_a(T[i + 1], s) + 128)
        return fail("packed word");
  }
  return 0;
}

// one dot product of K terms through digits, started FP32 accumulation in a
// random order (each step must be exact) and recombination
template <int K>
static int check_dot(int mode, double* worst) {
  double x[K], m[K];
  uint32_t mx = 0, mb = 0;
  for (int k = 0; k < K; ++k) {
    x[k] = mode == 1 ? -(2.0 - 0.008) : draw(mode == 2 ? 60 : 3);
    m[k] = mode == 1 ? -(2.0 - 0.008) : draw(mode == 2 ? 60 : 3);
    mx = std::max(mx, hi(x[k]) & 0x7FFFFFFFu);
    mb = std::max(mb, hi(m[k]) & 0x7FFFFFFFu);
  }
  const uint32_t ea = row_field(mx), eb = row_field(mb);
  std::vector<int> a(7 * K), b(8 * K);
  int colsum[8] = {0};
  for (int k = 0; k < K; ++k) {
    const uint64_t t = bytes_of(hi(x[k]), lo(x[k]), ea + 0x100000u);
    for (int s = 0; s < 7; ++s) a[s * K + k] = digit_a(t, s);
    int d[8];
    digits_b(hi(m[k]), lo(m[k]), eb, d);
    if (mode == 3)                               // extreme digits of one sign: the largest levels
      for (int s = 0; s < 8; ++s) {
        if (s < 7) a[s * K + k] = -128;
        d[s] = (k + s) % 5 ? -128 : 127;
      }
    for (int s = 0; s < 8; ++s) {
      if (d[s] < -128 || d[s] > 127) return fail("matrix digit range");
      b[s * K + k] = d[s];
      colsum[s] += d[s];
    }
    if (mode != 3) {
      i128 V = 0;
      for (int s = 0; s < 8; ++s) V = V * 256 + d[s];
      const long double want = std::ldexp((long double)m[k], 62 - ((int)(eb >> 20) - 1023));
      if (std::fabs((double)((long double)V - want)) > 0.5) return fail("matrix digit value");
    }
  }
  float v[8];
  i128 R = 0;
  for (int L = 0; L < 8; ++L) {
    const int P = start_value(L, K, colsum);
    int p[3];
    split_start(P, p);
    if (p[0] + 256 * p[1] + 65536 * p[2] != P || std::abs(p[0]) > 256 || std::abs(p[1]) > 256 || std::abs(p[2]) > 256)
      return fail("start split");
    std::vector<int> terms;
    long long level = 0;
    for (int s = 0; s < 7; ++s) {
      const int t = L - s;
      if (t < 0 || t > 7) continue;
      for (int k = 0; k < K; ++k) {
        terms.push_back((a[s * K + k] + 128) * b[t * K + k]);
        level += (long long)a[s * K + k] * b[t * K + k];
      }
    }
    for (size_t i = terms.size(); i > 1; --i) std::swap(terms[i - 1], terms[rng() % i]);
    float acc = std::ldexp((float)P, -24);
    long long exact = P;
    for (int q : terms) {
      acc += std::ldexp((float)q, -24);
      exact += q;
      if (mode != 3 && (double)acc != std::ldexp((double)exact, -24)) return fail("inexact accumulation");
      if (mode == 3 && std::llabs(exact) <= (1 << 24) && (double)acc != std::ldexp((double)exact, -24))
        return fail("inexact accumulation (extremes)");
    }
    if (std::llabs(level) > level_bound(L, K)) return fail("level bound");
    v[L] = acc;
    R = R * 256 + level;
  }
  const int64_t Q = combine<K>(v);
  const i128 want = (R + 32768) >> 16;
  const i128 diff = (i128)Q - want;
  if (diff > 1 || diff < -1 || (K <= 32 && mode != 3 && diff != 0)) return fail("recombination");
  if (mode == 3) return 0;
  // y against the exact sum (long double products, compensated): error in units of 2^(Ea + Eb - 52)
  long double y = 0.0L, c = 0.0L, sm = 0.0L;
  for (int k = 0; k < K; ++k) {
    const long double p = (long double)x[k] * (long double)m[k];
    const long double e = std::fmal(x[k], m[k], -p);
    const long double t = y + p;
    c += (std::fabs((double)y) >= std::fabs((double)p) ? (y - t) + p : (p - t) + y) + e;
    y = t;
    sm += std::fabs((double)m[k]);
  }
  y += c;
  const int Ea = (int)(ea >> 20) - 1023, Eb = (int)(eb >> 20) - 1023;
  const long double got = std::ldexp((long double)Q, Ea + Eb - kScale);
  // half a unit of V_a (plus truncated guard bits) per amplitude, half a unit of a
  // rounded matrix entry, Q's rounding, dropped products, low levels read short
  const long double bound = std::ldexp(sm, Ea - 54) * (0.5L + 1.0L / 256) +
                            K * std::ldexp(1.0L, Ea + 1) * std::ldexp(0.5L, Eb - 62) +
                            std::ldexp(0.5L + 0.02L + 6.0L * K / 1024, Ea + Eb - kScale);
  const double r = (double)(std::fabs((double)(got - y)) / bound);
  if (r > *worst) *worst = r;
  return r > 1.0 ? fail("dot product bound") : 0;
}

template <int K>
static int run(double* worst) {
  for (int i = 0; i < 4000; ++i)
    if (check_dot<K>(i % 4 == 3 ? (i % 8 == 3 ? 1 : 3) : i % 4, worst)) return 1;
  return 0;
}

int main() {
  for (int i = 0; i < 400000; ++i)
    if (check_row((int)(rng() % 80), (int)(rng() % 1600) - 800)) return 1;
  // zeros and subnormals in rows at the floor
  for (double x : {0.0, -0.0, 4.9e-324, -2.2e-308}) {
    const uint64_t t = bytes_of(hi(x), lo(x), ((uint32_t)kFloor << 20) + 0x100000u);
    for (int s = 0; s < kA; ++s)
      if (digit_a(t, s) != 0) return fail("zero or subnormal");
  }
  double worst = 0.0;
  if (run<8>(&worst) || run<16>(&worst) || run<32>(&worst) || run<64>(&worst) || run<128>(&worst)) return 1;
  printf("ok, worst dot product error %.3f of its bound\n", worst);
  return 0;
}
