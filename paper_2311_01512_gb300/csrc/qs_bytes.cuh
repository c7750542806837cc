// Byte slicing of FP64 operands for exact products on the fp16 tensor cores
// (the Ozaki scheme: Ozaki, Ogita, Oishi and Rump, "Error-free transformations
// of matrix multiplication by using fast routines of matrix multiplication and
// its applications", Numer. Algorithms 59 (2012)), with digits of radix 2^8.
//
// A matrix C = A B of K-term dot products: a row of A (amplitudes) and a column
// of B (gate matrix) are each scaled by a power of two, 2^E with |x| below
// (2 - 2^-7) 2^E, and cut into balanced digits -128 <= d <= 127:
//   V_a = x 2^(54 - Ea) rounded, |V_a| < 2^55: V_a = sum_{s<7} a_s 2^(8 (6 - s))
//   V_b = m 2^(62 - Eb) rounded, |V_b| < 2^63: V_b = sum_{t<8} b_t 2^(8 (7 - t))
// The products a_s b_t with L = s + t <= 7 are summed exactly, one accumulator
// per level L, and
//   y = Q 2^(Ea + Eb - 52 - X),  Q = round(sum_L level_L 2^(8 (7 - L)) / 2^(16 - X)),
// with X = 2 extra bits where they fit (K <= 64; |Q| < K 2^(54 + X)): a unit of Q is then
// one of V_a times a power-of-two matrix entry, and a row with one nonzero entry (a
// permutation, a diagonal) gives back what V_a holds: every bit of amplitudes within
// 2^-2 of the row's largest.
// Errors: half a unit of V_a per amplitude (2^-55 2^Ea), nothing from entries of
// B within 2^10 of their column's largest, half a unit of Q, and the dropped
// products (below 6 K 2^14 2^-24 2^X units of Q, 0.4 2^X for K = 64).
//
// Amplitude digits as bytes.  The integer V_a 2^8 is shifted into place with
// eight guard bits (truncated) and one 64-bit addition of 128 in every byte
// does both the rounding (byte 0) and the balancing: T = V_a 2^8 +
// 0x8080808080808080, byte 7 - s of T is a_s + 128.  No carry leaves byte 7,
// since |V_a| <= 2^55 - 2^47 - 2^40 by the bound on |x| above.  A byte f is the
// fp16 number f 2^-24 as it stands (a subnormal: the bit pattern f), so an
// operand word is two bytes and two zeros, moved by byte permutes.
//
// The offset 128 adds 128 sum_k b_t(k) to every level it meets; the accumulators
// start at minus that (P_L below), so that they end at level_L 2^-24.  Sums of
// any subset of a level's terms stay integers of at most (L + 1) 2^14 K <= 2^24
// (seven terms at L = 7), so FP32 accumulation is exact for K <= 128.  Levels of
// at most 2^22 also start at 0.75 = 1.5 2^23 2^-24 and end as the FP32 bit
// pattern 0x3F400000 + level.
//
// Host and device code (the host build is checked on the CPU).
#pragma once

#include <cstdint>

#include "qs_df.cuh"

namespace qsby {

constexpr int kA = 7;        // digits of an amplitude
constexpr int kB = 8;        // digits of a matrix entry
constexpr int kLevels = 8;   // levels kept
constexpr uint32_t kMagicBits = 0x3F400000u;   // 0.75
constexpr int kMagicInt = 12582912;            // 0.75 2^24
constexpr int kRoundQ = 32768;                 // half a unit of Q at X = 0, in units of level 7
constexpr int kScale = 52;                     // y = Q 2^(Ea + Eb - kScale - X)
QS_HD constexpr int extra_bits(int K) { return K <= 64 ? 2 : 0; }   // X

// Lower bound of a row's biased exponent: zeros and subnormals, whose implicit
// bit is wrongly set below, are then shifted below half a unit.
constexpr int kFloor = 58;

// Exponent field (biased exponent << 20) of a row or column whose largest
// high word without sign is mx: one more when its significand is 2 - 2^-7 or
// above (0x2080 / 2^20 = 0.00793), so that no digit sum carries out of T.
QS_HD uint32_t row_field(uint32_t mx) {
  const uint32_t e = (mx + 0x2080u) & 0x7FF00000u;
  return e > ((uint32_t)kFloor << 20) ? e : (uint32_t)kFloor << 20;
}

QS_HD uint64_t shr64(uint64_t x, uint32_t d) {
#if defined(__CUDA_ARCH__)
  uint64_t r;
  asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(d));   // amounts above 63 give 0
  return r;
#else
  return d > 63 ? 0ull : x >> d;
#endif
}

QS_HD uint32_t funnel_l(uint32_t lo, uint32_t hi, int s) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_l(lo, hi, s);
#else
  return (hi << s) | (lo >> (32 - s));
#endif
}

// T of the double hw:lw in a row of exponent field ef, ef1 = ef + 2^20.
QS_HD uint64_t bytes_of(uint32_t hw, uint32_t lw, uint32_t ef1) {
  const uint32_t sh = (ef1 - (hw & 0x7FF00000u)) >> 20;              // >= 1
  const uint64_t m = ((uint64_t)(funnel_l(lw, hw, 11) | 0x80000000u) << 32) | (lw << 11);
  const uint64_t sm = (uint64_t)(int64_t)((int32_t)hw >> 31);
  return (shr64(m, sh) ^ sm) - sm + 0x8080808080808080ull;
}

QS_HD int digit_a(uint64_t t, int s) { return (int)((t >> (8 * (7 - s))) & 255u) - 128; }

// byte i of the result is byte ((sel >> 4i) & 7) of the eight bytes (y:x)
QS_HD uint32_t perm(uint32_t x, uint32_t y, uint32_t sel) {
#if defined(__CUDA_ARCH__)
  return __byte_perm(x, y, sel);
#else
  const uint64_t v = ((uint64_t)y << 32) | x;
  uint32_t r = 0;
  for (int i = 0; i < 4; ++i) r |= (uint32_t)((v >> (8 * ((sel >> (4 * i)) & 7))) & 0xFF) << (8 * i);
  return r;
#endif
}

// The fp16 pairs (re in bits 0..15, im in 16..31) of all seven digits: two
// digits' bytes side by side in one permute, then a mask and a second permute.
QS_HD void packed_digits(uint64_t tre, uint64_t tim, uint32_t* w) {
  const uint32_t rl = (uint32_t)tre, rh = (uint32_t)(tre >> 32), il = (uint32_t)tim, ih = (uint32_t)(tim >> 32);
  const uint32_t p0 = perm(rh, ih, 0x6723u), p2 = perm(rh, ih, 0x4501u), p4 = perm(rl, il, 0x6723u);
  w[0] = p0 & 0x00FF00FFu;
  w[1] = perm(p0, 0u, 0x4341u);
  w[2] = p2 & 0x00FF00FFu;
  w[3] = perm(p2, 0u, 0x4341u);
  w[4] = p4 & 0x00FF00FFu;
  w[5] = perm(p4, 0u, 0x4341u);
  w[6] = perm(rl, il, 0x5511u) & 0x00FF00FFu;
}

// The eight digits of a matrix entry in a column of exponent field ef.
QS_HD void digits_b(uint32_t hw, uint32_t lw, uint32_t ef, int* d) {
  const uint32_t e = hw & 0x7FF00000u;
  const uint32_t sh = (ef - e) >> 20;
  uint64_t m = (((uint64_t)((hw & 0xFFFFFu) | 0x100000u) << 32) | lw) << 10;
  if (e == 0) m = 0;                                                 // zeros and subnormals
  if (sh > 0) m = sh > 63 ? 0ull : (m + (1ull << (sh - 1))) >> sh;
  // balanced as in T; |V_b| <= 2^63 - 2^55 - 2^48 by the bound on the entry, so nothing overflows
  const int64_t t = ((int32_t)hw < 0 ? -(int64_t)m : (int64_t)m) + 0x0080808080808080ll;
  d[0] = (int)(t >> 56);
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
  for (int k = 1; k < kB; ++k) d[k] = (int)((t >> (8 * (kB - 1 - k))) & 255) - 128;
}

// Largest |level L| (and |partial sum|) of K terms.
QS_HD constexpr int level_bound(int L, int K) { return (L < kA ? L + 1 : kA) * 16384 * K; }
QS_HD constexpr bool magic_level(int L, int K) { return level_bound(L, K) <= (1 << 22); }
// Levels 6 and 7 hold less than one unit of Q in their low bits: above 2^22 they
// are read divided by 2 or 4 (2^-5 of a unit of Q at X = 2).
QS_HD constexpr int low_shift(int K) { return level_bound(7, K) <= (1 << 22) ? 0 : (level_bound(7, K) <= (1 << 23) ? 1 : 2); }

// Start of level L: minus the offset's share, the magic where it fits, half a
// unit of Q in level 7.  colsum[t] = sum_k b_t(k).
QS_HD int start_value(int L, int K, const int* colsum, int X = 0) {
  int c = 0;
  for (int t = L < kA ? 0 : L - kA + 1; t <= L; ++t) c += colsum[t];
  return (magic_level(L, K) ? kMagicInt : 0) + (L == kLevels - 1 ? kRoundQ >> X : 0) - 128 * c;
}

// P = p[0] + 256 p[1] + 65536 p[2] with |p[i]| <= 256 (exact in fp16), for
// |P| <= 2^24: the initialising MMA multiplies them by 2^-24, 2^-16 and 2^-8.
QS_HD void split_start(int P, int* p) {
  p[2] = (P + (P >= 0 ? 32768 : -32768)) / 65536;
  const int r = P - 65536 * p[2];
  p[1] = (r + (r >= 0 ? 128 : -128)) / 256;
  p[0] = r - 256 * p[1];
}

// A result is Q as a double times 2^(inc / 2^20).  Adding inc to the exponent field
// does it where no nonzero Q (1 <= |Q| < 2^62) leaves the normal numbers:
constexpr int kMinInc = -(1022 << 20), kMaxInc = (2046 - 1023 - 62) << 20;
QS_HD double add_inc(double r, int inc) {
  uint32_t hw, lw;
  qsdf::d2w(r, hw, lw);                          // hw is 0 only for r = 0, which stays 0
  return qsdf::w2d(hw != 0 ? hw + (uint32_t)inc : 0u, lw);
}
// Elsewhere two factors (|inc| < 2^31, so both are normal numbers): the first product
// is exact where the result is below it, so the result is rounded once, to a subnormal
// number, 0 or infinity where it has to be.
QS_HD double mul_inc(double r, int inc) {
  const int e = inc >> 20, e1 = e / 2;
  return r * qsdf::w2d((uint32_t)(1023 + e1) << 20, 0u) * qsdf::w2d((uint32_t)(1023 + e - e1) << 20, 0u);
}

QS_HD uint32_t fbits(float v) { return qsdf::f2u(v); }
QS_HD int to_int(float v) { return (int)v; }   // exact integers

// Q from the accumulators v_L.  Magic levels hold 0x3F400000 + level in their
// bits; r = 256 b_L + b_(L+1) is then 0x7F400000 + 256 level_L + level_(L+1)
// mod 2^32, without a wrap for levels of at most 2^22 (257 2^22 < 0x7F400000),
// so the offsets leave as constants.
template <int K, int X = 0>
QS_HD int64_t combine(const float* v) {
  constexpr uint32_t off = 0x7F400000u;
  const uint32_t r0 = fbits(v[0]) * 256u + fbits(v[1]);
  if constexpr (K <= 32) {
    const uint32_t r1 = fbits(v[2]) * 256u + fbits(v[3]), r2 = fbits(v[4]) * 256u + fbits(v[5]);
    const uint32_t r3 = fbits(v[6]) * 256u + fbits(v[7]);
    constexpr uint64_t C = ((((uint64_t)off << 32) + ((uint64_t)off << 16) + off) << X) + (off >> (16 - X));
    return (int64_t)(((uint64_t)r0 << (32 + X)) + ((uint64_t)r1 << (16 + X)) + ((uint64_t)r2 << X) +
                     (uint64_t)(r3 >> (16 - X)) - C);
  } else {
    constexpr int ls = low_shift(K);
    constexpr float lf = ls == 1 ? 0.5f : 0.25f;
    const uint32_t b6 = fbits(qsdf::fmaf_(v[6], lf, 0.75f)), b7 = fbits(qsdf::fmaf_(v[7], lf, 0.75f));
    const uint32_t r3 = b6 * 256u + b7;
    if constexpr (K <= 64) {                       // levels 4 and 5 above 2^22: as integers plus 2^23
      const uint32_t r1 = fbits(v[2]) * 256u + fbits(v[3]);
      const uint32_t l4 = (uint32_t)to_int(qsdf::fmaf_(v[4], 16777216.0f, 8388608.0f));
      const uint32_t l5 = (uint32_t)to_int(qsdf::fmaf_(v[5], 16777216.0f, 8388608.0f));
      const uint32_t r2 = l4 * 256u + l5;
      constexpr uint64_t C = ((((uint64_t)off << 32) + ((uint64_t)off << 16) + 257ull * 8388608ull) << X) +
                             (off >> (16 - ls - X));
      return (int64_t)(((uint64_t)r0 << (32 + X)) + ((uint64_t)r1 << (16 + X)) + ((uint64_t)r2 << X) +
                       (uint64_t)(r3 >> (16 - ls - X)) - C);
    } else {                                       // levels 2 to 5
      static_assert(X == 0, "no room for more bits");
      const int32_t q1 = to_int(v[2] * 16777216.0f) * 256 + to_int(v[3] * 16777216.0f);
      const int64_t q2 = (int64_t)to_int(v[4] * 16777216.0f) * 256 + to_int(v[5] * 16777216.0f);
      constexpr uint64_t C = ((uint64_t)off << 32) + (off >> (16 - ls));
      return (int64_t)(((uint64_t)r0 << 32) + (uint64_t)((int64_t)q1 * 65536) + (uint64_t)q2 +
                       (uint64_t)(r3 >> (16 - ls)) - C);
    }
  }
}

}  // namespace qsby
