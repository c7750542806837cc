// Host check of the output scaling of the byte-slice kernels (qs_bytes.cuh): adding
// an increment to the exponent field inside its limits and multiplying outside them,
// against ldexp, from the smallest results to the largest.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

#include "qs_bytes.cuh"

static bool same(double a, double b) { return std::memcmp(&a, &b, 8) == 0; }

int main() {
  std::mt19937_64 rng(11);
  for (int e = -1982; e <= 1996; ++e)
    for (int i = 0; i < 400; ++i) {
      int64_t q = (int64_t)(rng() >> (2 + rng() % 62));          // below 2^62
      if (i == 0) q = 0;
      if (i == 1) q = 1;
      if (i == 2) q = (1ll << 62) - 1;
      const double r = (double)(i & 1 ? -q : q), want = std::ldexp(r, e);
      const int inc = e * (1 << 20);
      if (q == 0 && qsby::mul_inc(0.0, inc) != 0.0) return std::printf("zero, e = %d\n", e), 1;
      if (q != 0 && !same(qsby::mul_inc(r, inc), want)) return std::printf("mul_inc(%a, %d)\n", r, e), 1;
      if (inc >= qsby::kMinInc && inc <= qsby::kMaxInc && qsby::add_inc(r, inc) != want)
        return std::printf("add_inc(%a, %d)\n", r, e), 1;
    }
  std::printf("ok\n");
  return 0;
}
