// Host program for the dense gates of small statevectors in block fixed point
// (k_dense_fx, qs_gates_fx.cu): reads rows from stdin and prints the real part that
// the kernel computes for them, so that the Python test can compare with exact
// rational arithmetic.
//
// Input, one row per line (64-bit patterns of doubles in hex):
//   NT  x_0.re x_0.im ..  m_0.re m_0.im ..     (2^NT complex numbers each)
// Output, one line per row: the pattern of Re sum_k m_k x_k.
#include <cinttypes>
#include <cstdio>
#include <cstring>

#include "qs_fx.cuh"

int main() {
  int nt;
  while (std::scanf("%d", &nt) == 1) {
    if (nt < 2 || nt > 5) return 2;
    const int D = 1 << nt, SH = nt - 2;
    double x[64], m[64];
    for (int k = 0; k < 4 * D; ++k) {
      uint64_t u;
      if (std::scanf("%" SCNx64, &u) != 1) return 2;
      std::memcpy(k < 2 * D ? x + k : m + (k - 2 * D), &u, 8);
    }
    int ex = 0, em = 0;
    for (int k = 0; k < 2 * D; ++k) {
      ex = ex > qsfx::expo_of(x[k]) ? ex : qsfx::expo_of(x[k]);
      em = em > qsfx::expo_of(m[k]) ? em : qsfx::expo_of(m[k]);
    }
    int64_t v = 0;
    for (int k = 0; k < D; k += 2) {
      qsfx::Acc a = qsfx::acc_zero();
      for (int u = k; u < k + 2; ++u) {
        const qsfx::Part xr = qsfx::fixed_d(x[2 * u], ex), xi = qsfx::fixed_d(x[2 * u + 1], ex);
        qsfx::mac(a, xr, qsfx::fixed_const(m[2 * u], em));
        qsfx::mac(a, qsfx::Part{-xi.h, -xi.l}, qsfx::fixed_const(m[2 * u + 1], em));
      }
      v += qsfx::partial(a, SH);
    }
    const double y = qsfx::finish_v(v, qsfx::scale_for(ex + SH, em));
    uint64_t u;
    std::memcpy(&u, &y, 8);
    std::printf("%016" PRIx64 "\n", u);
  }
  return 0;
}
