// Superoperators of one- and two-qubit Kraus maps, formed on the host (no CUDA
// dependency, so the host check tests/host/superop1_check.cpp compiles it
// with g++ alone).
#pragma once

#include <cmath>

namespace qsh {

// sum_m conj(K_m) (x) K_m of one-qubit operators K_m (row-major 2x2, re/im
// interleaved) as a 4x4 matrix (Sec. "Kraus map"): row r = 2 i + k, column
// c = 2 j + l, entry sum_m conj(K_m[i][j]) K_m[k][l]; index bit 0 acts on the
// ket qubit t, bit 1 on the bra qubit t + N.  The same entries as the device
// superoperator kernel; the library makes the block fixed-point constants of
// a one-pass Kraus map from it.  sup: 32 doubles (16 complex, row-major).
inline void superop1(const double* kraus, int num_ops, double* sup) {
  for (int e = 0; e < 32; ++e) sup[e] = 0.0;
  for (int m = 0; m < num_ops; ++m) {
    const double* K = kraus + 8 * m;
    for (int r = 0; r < 4; ++r)
      for (int c = 0; c < 4; ++c) {
        const int a = 2 * (r >> 1) + (c >> 1), b = 2 * (r & 1) + (c & 1);
        const double ar = K[2 * a], ai = -K[2 * a + 1], br = K[2 * b], bi = K[2 * b + 1];
        sup[2 * (4 * r + c)] += ar * br - ai * bi;
        sup[2 * (4 * r + c) + 1] += ar * bi + ai * br;
      }
  }
}

// The same of two-qubit operators (4x4) as a 16x16 matrix, row 4 i + k, column
// 4 j + l, with the operations of the device superoperator kernel one by one (a
// fused multiply-add on a product, operators added in order), so that both
// give the same bits.  sup: 512 doubles (256 complex, row-major).
inline void superop2(const double* kraus, int num_ops, double* sup) {
  for (int e = 0; e < 512; ++e) sup[e] = 0.0;
  for (int m = 0; m < num_ops; ++m) {
    const double* K = kraus + 32 * m;
    for (int i = 0; i < 4; ++i)
      for (int k = 0; k < 4; ++k)
        for (int j = 0; j < 4; ++j) {
          const double ar = K[2 * (4 * i + j)], ai = -K[2 * (4 * i + j) + 1];
          double* out = sup + 2 * (16 * (4 * i + k) + 4 * j);
          for (int l = 0; l < 4; ++l) {
            const double br = K[2 * (4 * k + l)], bi = K[2 * (4 * k + l) + 1];
            out[2 * l] += std::fma(ar, br, -(ai * bi));
            out[2 * l + 1] += std::fma(ar, bi, ai * br);
          }
        }
  }
}

}  // namespace qsh
