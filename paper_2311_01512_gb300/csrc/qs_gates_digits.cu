// Dense gates on the Choi vector of a small density matrix in exact 7-bit digits
// (qs_slices.cuh) on the CUDA cores.
//
// The update alpha_kj -> sum_l m_jl alpha_kl (Sec. "Many-target gate", Eq. (local
// many-target amplitude update)) with each group of 2^NT amplitudes cut into
// eight balanced digits under its largest exponent and each column of the
// realified matrix under its own; the digit products with s + t <= 7 summed per
// level s + t, recombined in integers, rounded down to a multiple of 2^-53 of the two
// scales and then to double.  With Ea, Eb the exponents of the group's and the column's
// largest parts and K = 2^(NT + 1) real terms, an error of at most
//   2^-53 |y| + (K + 1) 2^-53 2^(Ea + Eb)   (tests/host/slices_check.cpp),
// measured 7e-17 of the outputs' rms on dense rows.
// Why not block fixed point, as for statevectors (2.7 us where this takes 4.3): Pauli sums
// over small noisy density matrices cancel, in some to a small part of their terms, and a
// change of rounding in the operations before moved 3 of 60 such sums by more than the
// 8e-15 that they are held to.  Larger density matrices take the byte slices
// (qs_tc_ozaki.cu), which round otherwise.
//
// Work mapping: two threads per amplitude, one for each part of the output.
// Thread (group, part c, j) slices part c of amplitude j; the block's digits and
// the matrix digits (of re, im and -im) go through shared memory as floats, and
// every product is an FMA on integers below 2^24, exact in any order.  36 FMAs
// per real multiply-add, 128 a clock and SM: about 1200 issue slots a thread for
// four targets, against a setup of some 300.
// Why: on 4096 amplitudes the tensor-core kernel ran two tiles on two SMs behind
// a setup that slices the whole matrix.  4096 amplitudes, four targets, us a
// pass in a replayed program: 10.9 -> 4.3.
#include <cstring>

#include "qs_bytes.cuh"
#include "qs_device.cuh"
#include "qs_slices.cuh"

namespace qsk {
namespace {

constexpr int kDigitThreads = 128;
constexpr int kExpFloor = 58;     // zeros and subnormals shift out entirely

// digits of x under the biased exponent em, as 8 floats at two 16-byte words hstride floats apart
__device__ __forceinline__ void put_digits(float* dst, int hstride, double x, int em) {
  float f[8];
  qsoz::digit_floats_t8(qsoz::fixed_t8((uint32_t)__double2hiint(x), (uint32_t)__double2loint(x), em), f);
  *reinterpret_cast<float4*>(dst) = make_float4(f[0], f[1], f[2], f[3]);
  *reinterpret_cast<float4*>(dst + hstride) = make_float4(f[4], f[5], f[6], f[7]);
}

__device__ __forceinline__ void get_digits(const float* src, int hstride, float* f) {
  const float4 a = *reinterpret_cast<const float4*>(src), b = *reinterpret_cast<const float4*>(src + hstride);
  f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
  f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}

__device__ __forceinline__ int exp_of(double x) { return qsoz::biased_exp((uint32_t)__double2hiint(x)); }

template <int NT>
struct DigitSmem {
  static constexpr int D = 1 << NT, G = kDigitThreads / (2 * D);   // groups per block
  static constexpr int XF = kDigitThreads * 8;                     // amplitude digits: [group][k][part][8]
  static constexpr int MF = D * 3 * 2 * D * 4;                     // matrix digits: [k][re, im, -im][half][j][4]
  static constexpr size_t bytes = 4 * (size_t)(XF + MF + D + G);
};

}  // namespace

template <int NT, typename Mat>
__global__ void __launch_bounds__(kDigitThreads) k_dense_digits(double2* __restrict__ psi,
                                                                const __grid_constant__ DenseFxParams p,
                                                                const __grid_constant__ Mat mat) {
  using S = DigitSmem<NT>;
  constexpr int D = S::D;
  extern __shared__ __align__(16) float sm[];
  float* xd = sm;
  float* md = xd + S::XF;
  int* cexp = reinterpret_cast<int*>(md + S::MF);   // D: column exponents (both parts of output j share one)
  int* rexp = cexp + D;                             // G: row exponents
  const int tid = threadIdx.x, j = tid % D, c = (tid / D) & 1, gi = tid / (2 * D);
  const uint64_t k0 = (uint64_t)blockIdx.x * S::G + gi;
  const bool ok = k0 < p.ngroups;
  uint64_t i = insert_zeros(k0, p.ins, p.nins) | p.ctrl_mask;
#pragma unroll
  for (int q = 0; q < NT; ++q)
    if ((j >> q) & 1) i |= 1ull << p.tpos[q];
  const double2 a = ok ? psi[i] : make_double2(0.0, 0.0);
  constexpr int E = (D * D + kDigitThreads - 1) / kDigitThreads;   // matrix entries per thread
  double2 m[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int idx = tid + e * kDigitThreads, row = idx / D, l = idx % D, mm = (1 << p.nmat) - 1;
    m[e] = make_double2(0.0, 0.0);
    // an identity on the targets beyond the stored matrix
    if (idx < D * D && (row >> p.nmat) == (l >> p.nmat))
      m[e] = mat.m[((row & mm) << p.nmat) + (l & mm)];
    if (p.conj) m[e].y = -m[e].y;
  }
  for (int n = tid; n < D; n += kDigitThreads) cexp[n] = kExpFloor;
  if (tid < S::G) rexp[tid] = kExpFloor;
  __syncthreads();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int idx = tid + e * kDigitThreads;
    if (idx < D * D) atomicMax(cexp + idx / D, max(exp_of(m[e].x), exp_of(m[e].y)));
  }
  const double own = c ? a.y : a.x;
  atomicMax(rexp + gi, exp_of(own));
  __syncthreads();
  const int er = rexp[gi];
  put_digits(xd + ((gi * D + j) * 2 + c) * 8, 4, own, er);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int idx = tid + e * kDigitThreads, row = idx / D, l = idx % D;
    if (idx < D * D) {
      float* dst = md + l * (6 * D * 4) + row * 4;
      put_digits(dst, D * 4, m[e].x, cexp[row]);
      put_digits(dst + 2 * D * 4, D * 4, m[e].y, cexp[row]);
      put_digits(dst + 4 * D * 4, D * 4, -m[e].y, cexp[row]);
    }
  }
  __syncthreads();
  // re: xr mr + xi (-mi); im: xr mi + xi mr.  Levels start at the magic that
  // leaves their integers in the bit pattern (sums of at most 2.5 2^20).
  float lv[8];
#pragma unroll
  for (int L = 0; L < 8; ++L) lv[L] = 12582912.0f;
  const float* xg = xd + gi * D * 16;
  const float* m0 = md + (c ? 2 * D * 4 : 0) + j * 4;        // against xr
  const float* m1 = md + (c ? 0 : 4 * D * 4) + j * 4;        // against xi
#pragma unroll 2
  for (int k = 0; k < D; ++k) {
    float x[8], y[8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      get_digits(xg + k * 16 + h * 8, 4, x);
      get_digits((h ? m1 : m0) + k * (6 * D * 4), D * 4, y);
#pragma unroll
      for (int s = 0; s < 8; ++s)
#pragma unroll
        for (int t = 0; t + s < 8; ++t) lv[s + t] = fmaf(x[s], y[t], lv[s + t]);
    }
  }
  uint32_t bits[8];
#pragma unroll
  for (int L = 0; L < 8; ++L) bits[L] = __float_as_uint(lv[L]);
  const double r = __ll2double_rn(qsoz::combine_pairs_u<8, qsoz::kFaddMagicBits>(bits));
  const int inc = (er + cexp[j] - 2046 - 53) * (1 << 20);
  const bool rare = inc < qsby::kMinInc || inc > qsby::kMaxInc;
  const double o = rare ? qsby::mul_inc(r, inc) : qsby::add_inc(r, inc);
  if (ok) reinterpret_cast<double*>(psi)[2 * i + c] = o;
}

template <int NT, typename Mat>
static cudaError_t dense_digits(void* amps, const DenseFxParams& p, const Mat& mat, cudaStream_t st) {
  static bool attr_done = false;
  if (!attr_done) {
    const cudaError_t e = cudaFuncSetAttribute(k_dense_digits<NT, Mat>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)DigitSmem<NT>::bytes);
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  const unsigned g = (unsigned)((p.ngroups + DigitSmem<NT>::G - 1) / DigitSmem<NT>::G);
  k_dense_digits<NT, Mat><<<g, kDigitThreads, DigitSmem<NT>::bytes, st>>>(static_cast<double2*>(amps), p, mat);
  return cudaGetLastError();
}

template <int NT>
static cudaError_t dense_digits_n(void* amps, const DenseFxParams& p, const double* host_mat, cudaStream_t st) {
  if (!host_mat) return dense_digits<NT>(amps, p, MatPtr{reinterpret_cast<const double2*>(p.mat)}, st);
  MatArg<NT> m;
  std::memcpy(&m, host_mat, sizeof(double2) << (2 * p.nmat));
  return dense_digits<NT>(amps, p, m, st);
}

cudaError_t launch_dense_digits(void* amps, const DenseFxParams& p, const double* host_mat, cudaStream_t st) {
  switch (p.n) {
    case 3: return dense_digits_n<3>(amps, p, host_mat, st);
    case 4: return dense_digits_n<4>(amps, p, host_mat, st);
    case 5: return dense_digits_n<5>(amps, p, host_mat, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qsk
