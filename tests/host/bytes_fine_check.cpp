// Host check of the recombination with extra bits (csrc/qs_bytes.cuh, K <= 64 terms):
// against 128-bit integers, and the error of whole dot products of rows with one nonzero
// entry (permutations, diagonals) and of dense rows.  Prints, per K, the rms and the mean
// error of one-entry rows in units of the row's largest amplitude and the rms error of
// dense rows in units of the results' rms.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

#include "qs_bytes.cuh"

using namespace qsby;
typedef __int128 i128;

static uint32_t hi(double x) { uint64_t u; memcpy(&u, &x, 8); return (uint32_t)(u >> 32); }
static uint32_t lo(double x) { uint64_t u; memcpy(&u, &x, 8); return (uint32_t)u; }
static int fail(const char* what) { printf("FAIL %s\n", what); return 1; }

template <int K>
static int run(std::mt19937_64& rng) {
  constexpr int X = extra_bits(K);
  std::normal_distribution<double> nd;
  double e2[2] = {0, 0}, mean = 0, y2 = 0;
  const int N = 60000;
  for (int it = 0; it < 2 * N; ++it) {
    const bool dense = it & 1;
    double x[K], m[K], norm = 0;
    for (int k = 0; k < K; ++k) {
      x[k] = nd(rng) * (rng() % 4 ? 1.0 : std::ldexp(1.0, -(int)(rng() % 12)));
      m[k] = nd(rng);
      norm += m[k] * m[k];
    }
    for (int k = 0; k < K; ++k) m[k] = dense ? m[k] / std::sqrt(norm) : 0.0;
    const int one = (int)(rng() % K);
    if (!dense) m[one] = rng() % 2 ? 1.0 : -1.0;
    uint32_t mx = 0, mb = 0;
    double row = 0;
    for (int k = 0; k < K; ++k) {
      mx = std::max(mx, hi(x[k]) & 0x7FFFFFFFu);
      mb = std::max(mb, hi(m[k]) & 0x7FFFFFFFu);
      row = std::max(row, std::fabs(x[k]));
    }
    const uint32_t ea = row_field(mx), eb = row_field(mb);
    int a[7][K], b[8][K], colsum[8] = {0};
    for (int k = 0; k < K; ++k) {
      const uint64_t t = bytes_of(hi(x[k]), lo(x[k]), ea + 0x100000u);
      for (int s = 0; s < 7; ++s) a[s][k] = digit_a(t, s);
      int d[8];
      digits_b(hi(m[k]), lo(m[k]), eb, d);
      for (int s = 0; s < 8; ++s) {
        b[s][k] = d[s];
        colsum[s] += d[s];
      }
    }
    float v[8];
    i128 R = 0;
    for (int L = 0; L < 8; ++L) {
      long long acc = start_value(L, K, colsum, X), level = 0;
      for (int s = 0; s < 7 && s <= L; ++s)
        for (int k = 0; k < K; ++k) {
          acc += (long long)(a[s][k] + 128) * b[L - s][k];
          level += (long long)a[s][k] * b[L - s][k];
        }
      v[L] = std::ldexp((float)acc, -24);
      if ((double)v[L] != std::ldexp((double)acc, -24)) return fail("level not exact");
      R = R * 256 + level;
    }
    const int64_t Q = combine<K, X>(v);
    const i128 want = (R + (32768 >> X)) >> (16 - X), diff = (i128)Q - want;
    if (diff > 1 || diff < -1 || (K <= 32 && diff != 0)) return fail("recombination");
    const int Ea = (int)(ea >> 20) - 1023, Eb = (int)(eb >> 20) - 1023;
    const double y = std::ldexp((double)Q, Ea + Eb - kScale - X);
    long double exact = 0;
    for (int k = 0; k < K; ++k) exact += (long double)x[k] * (long double)m[k];
    const double e = (double)((long double)y - exact);
    if (dense) {
      e2[1] += e * e;
      y2 += (double)(exact * exact);
    } else {
      const int held = (int)(hi(x[one]) >> 20 & 0x7FFu) - 1023;
      if (held >= Ea - 2 && e != 0.0) return fail("a large amplitude lost bits");
      if (std::fabs(e) > std::ldexp(0.5 + 1.0 / 256, Ea - 54)) return fail("a small amplitude beyond half a unit");
      e2[0] += e / row * (e / row);
      mean += e / row;
    }
  }
  std::printf("%d %.4g %.4g %.4g\n", K, std::sqrt(e2[0] / N), mean / N, std::sqrt(e2[1] / y2));
  return 0;
}

int main() {
  std::mt19937_64 rng(19);
  return run<16>(rng) || run<32>(rng) || run<64>(rng);
}
