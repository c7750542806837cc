// Dense n-target gates (2 <= n <= 6) for complex128 states on the fp16 tensor
// cores, with error-free byte slicing (the Ozaki scheme; the slicing, its bounds
// and the recombination are in qs_bytes.cuh).
//
// The group update alpha_kj -> sum_l m_jl alpha_kl (Sec. "Many-target gate",
// Eq. (local many-target amplitude update)) over a tile of 128 groups is the
// real GEMM C = A B, A[g, 2l + c'] the interleaved (re, im) amplitudes of group
// g, B the realified matrix (B[2l, 2j] = Re m_jl, B[2l+1, 2j] = -Im m_jl,
// B[2l, 2j+1] = Im m_jl, B[2l+1, 2j+1] = Re m_jl).  Each row of A (scaled by
// its largest exponent) is cut into seven balanced bytes and each column of B
// into eight; the 35 slice products with s + t <= 7 run as tcgen05 kind::f16
// MMAs whose FP32 accumulation in tensor memory is exact, one accumulator per
// level L = s + t; the epilogue recombines the levels in integers, converts
// once to double and applies the two scales.  Two targets run as three: the
// matrix is extended by an identity on one more (free) qubit, which changes
// nothing in the result and fills the MMA's K = 16.
//
// The amplitude bytes are stored with an offset of 128 as fp16 subnormals.
// Each tile's accumulators start at P_L(n), minus the offset's contribution
// (plus the magic that leaves a level's integer in the low bits of its FP32
// pattern, where it fits).  One initialising MMA writes them: a constant A
// whose rows are (2^-24, 2^-16, 2^-8, 0, ...) against a B whose column holds
// P = p0 + 256 p1 + 65536 p2 in three fp16-exact parts.
//
// Why bytes: the kernels are bound by the integer pipe (a byte permute or a
// logic operation per digit and pair, 64 a clock and SM), so what counts is the
// integer instructions per amplitude.  Balanced 7-bit digits in bf16 (eight a
// side) took about 95; byte-aligned digits need no shift per digit, no separate
// top digit, one addition for rounding and balancing, and about 65.
// Measured at 28 qubits, spread targets, per pass (the copy rate would take 1.27
// ms): 3 targets 1.95 -> 1.50 ms, 4 targets 1.94 -> 1.50, 5 targets 3.32 -> 2.30,
// 6 targets (native FP64 before) 110.6 -> 4.0 with a matrix that mixes its groups (any
// other stays in FP64, see k_wide_matrix).  Against extended precision the relative
// error of an output vector is 5.4, 5.4, 5.6 and 6.4e-17 (7-bit digits 7.7, 6.6 and 7.6,
// FP64 at six targets 37.5).
//
// Three kernels share these pieces: k_dense_ozaki_ws (two to four targets) and
// k_dense_ozaki5 give gathering and slicing, MMA issue and the epilogue to
// separate warps; k_dense_ozaki6 walks blocks of its product with the tile's
// amplitudes in registers.  Passes over few amplitudes go to k_dense_fx
// (qs_gates_fx.cu) instead, except with six targets.
#include "qs_device.cuh"
#include "qs_bytes.cuh"
#include "qs_tc_ptx.cuh"

namespace qsk {
namespace {

using namespace tcptx;

constexpr int kRows = 128;
constexpr uint32_t kWaitLimit = 1u << 26;

constexpr int kLv = qsby::kLevels;

// fp16 bit pattern of a small integer
__device__ __forceinline__ uint16_t half_bits(int v) {
  uint16_t r;
  asm("cvt.rn.f16.f32 %0, %1;" : "=h"(r) : "f"((float)v));
  return r;
}

// bounded wait on an mbarrier phase; true when it ran out
__device__ __forceinline__ bool wait_phase(uint64_t* bar, uint32_t parity) {
  uint32_t spins = 0;
  while (!mbar_try_wait(bar, parity))
    if (++spins > kWaitLimit) return true;
  return false;
}

// entry (j, l) of the complex (and possibly identity-extended) matrix, D x D
__device__ __forceinline__ double2 matrix_entry(const TcParams& p, int D, int jk, int lk) {
  int j = 0, l = 0;                               // kernel targets -> matrix bits
  for (int q = 0; q < p.n; ++q) {
    j |= (jk >> q & 1) << p.mbit[q];
    l |= (lk >> q & 1) << p.mbit[q];
  }
  if (p.nmat < p.n) {
    if ((j >> p.nmat) != (l >> p.nmat)) return make_double2(0.0, 0.0);
    const int mm = (1 << p.nmat) - 1;
    j &= mm;
    l &= mm;
    D = 1 << p.nmat;
  }
  double2 m = reinterpret_cast<const double2*>(p.mat)[j * D + l];
  if (p.conj) m.y = -m.y;
  return m;
}

__device__ __forceinline__ uint32_t abs_hi(double x) { return (uint32_t)__double2hiint(x) & 0x7FFFFFFFu; }

// The slices of B from the complex matrix: entry (j, l) = (re, im) gives rows 2l,
// 2l + 1 of column 2j (re, -im) and of column 2j + 1 (im, re), whose scales are
// one, so two sets of digits and 16 stores of a pair serve four entries (a
// negated digit stays within 128).  Leaves the column scales in csc and the digit
// column sums in colsum (2D x 8).  off(n, k): byte offset of entry (k, n) in a
// slice; slices are tstride bytes apart.  Ends with a barrier.
template <int NT, int NTHR, typename Off>
__device__ __forceinline__ void slice_matrix(const TcParams& p, unsigned char* b_dig, uint32_t tstride, const Off& off,
                                             int* csc, int* colsum, int tid) {
  constexpr int D = 1 << NT, E = (D * D + NTHR - 1) / NTHR;
  for (int n = tid; n < 2 * D; n += NTHR) csc[n] = 0;
  for (int i = tid; i < kLv * 2 * D; i += NTHR) colsum[i] = 0;
  __syncthreads();
  double2 m[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    // column fastest across threads: the lanes of a warp update different columns
    const int idx = tid + e * NTHR, j = idx % D, l = idx / D;
    if (idx >= D * D) break;
    m[e] = matrix_entry(p, D, j, l);
    atomicMax(csc + 2 * j, (int)max(abs_hi(m[e].x), abs_hi(m[e].y)));
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int idx = tid + e * NTHR, j = idx % D, l = idx / D;
    if (idx >= D * D) break;
    const uint32_t ef = qsby::row_field((uint32_t)csc[2 * j]);
    int dr[qsby::kB], di[qsby::kB];
    qsby::digits_b((uint32_t)__double2hiint(m[e].x), (uint32_t)__double2loint(m[e].x), ef, dr);
    qsby::digits_b((uint32_t)__double2hiint(m[e].y), (uint32_t)__double2loint(m[e].y), ef, di);
    unsigned char *b0 = b_dig + off(2 * j, 2 * l), *b1 = b_dig + off(2 * j + 1, 2 * l);
#pragma unroll
    for (int t = 0; t < qsby::kB; ++t) {
      const uint32_t hr = half_bits(dr[t]), hi = half_bits(di[t]);
      *reinterpret_cast<uint32_t*>(b0 + t * tstride) = hr | ((di[t] ? hi ^ 0x8000u : 0u) << 16);
      *reinterpret_cast<uint32_t*>(b1 + t * tstride) = hi | (hr << 16);
      atomicAdd(colsum + 2 * j * kLv + t, dr[t] - di[t]);
      atomicAdd(colsum + (2 * j + 1) * kLv + t, dr[t] + di[t]);
    }
  }
  __syncthreads();
}

// All slice products of one tile.  B's slices lie back to back in shared
// memory (slice t at t * bbytes), so for A slice s one MMA against the first
// 8 - s slices of B, with its accumulator starting at level s, adds A_s B_t
// into level s + t for every t <= 7 - s at once: each A slice is read once
// per 16-column K chunk.  Products wider than 256 columns are cut into
// 256-column MMAs.  adesc / bdesc: descriptors of slice 0 of A and B; K chunks
// are 256 bytes apart, 8-row groups of B kdim * 16 bytes (encoded address >> 4).
template <int N, int KCH>
__device__ __forceinline__ void mma_tile(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc) {
  constexpr int K = 16 * KCH;
  constexpr uint32_t abytes = kRows * K * 2;
#pragma unroll
  for (int s = 0; s < qsby::kA; ++s) {
    constexpr int kMax = 256;
#pragma unroll
    for (int c0 = 0; c0 < (kLv - s) * N; c0 += kMax) {
      const int w = (kLv - s) * N - c0 < kMax ? (kLv - s) * N - c0 : kMax;
      const uint32_t idesc = idesc_f16(kRows, w);
#pragma unroll
      for (int kk = 0; kk < KCH; ++kk)
        mma_f16(d_tmem + (uint32_t)(s * N + c0), adesc + ((s * abytes + kk * 256) >> 4),
                bdesc + (((uint32_t)c0 * K * 2 + kk * 256) >> 4), idesc, 1u);
    }
  }
}

// The initialising MMA: every level column of the buffer at dcol starts at its P_L(n).
template <int N>
__device__ __forceinline__ void mma_start(uint32_t dcol, const unsigned char* a_pre, const unsigned char* b_pre) {
  constexpr uint32_t LCOLS = kLv * N;
  const uint64_t pad = smem_desc(smem_u32(a_pre), 128, 256), pbd = smem_desc(smem_u32(b_pre), 128, 256);
#pragma unroll
  for (uint32_t c0 = 0; c0 < LCOLS; c0 += 256) {
    const uint32_t w = LCOLS - c0 < 256 ? LCOLS - c0 : 256;
    mma_f16(dcol + c0, pad, pbd + ((c0 * 32) >> 4), idesc_f16(kRows, (int)w), 0u);
  }
}

// Slice products of operands with K = 16 KCH columns.
template <int N, int KCH>
__device__ __forceinline__ void mma_products(uint32_t dcol, const unsigned char* A, const unsigned char* B) {
  constexpr uint32_t sbo = KCH * 16 * 16;
  mma_tile<N, KCH>(dcol, smem_desc(smem_u32(A), 128, sbo), smem_desc(smem_u32(B), 128, sbo));
}

// Rows (2^-24, 2^-16, 2^-8, 0, ...) of the initialising MMA's A: two 16-byte core-matrix rows each.
__device__ __forceinline__ void fill_start_rows(unsigned char* a_pre, int tid, int nthr) {
  for (int g = tid; g < kRows; g += nthr) {
    *reinterpret_cast<uint4*>(a_pre + canon_off16(g, 0, 16)) = make_uint4(0x01000001u, 0x1C00u, 0u, 0u);
    *reinterpret_cast<uint4*>(a_pre + canon_off16(g, 8, 16)) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// The column of the initialising MMA's B that starts level column `col` at P.
__device__ __forceinline__ void fill_start_column(unsigned char* b_pre, int col, int P) {
  int pp[3];
  qsby::split_start(P, pp);
  const uint32_t lo = half_bits(pp[0]) | ((uint32_t)half_bits(pp[1]) << 16);
  *reinterpret_cast<uint4*>(b_pre + canon_off16(col, 0, 16)) = make_uint4(lo, half_bits(pp[2]), 0u, 0u);
  *reinterpret_cast<uint4*>(b_pre + canon_off16(col, 8, 16)) = make_uint4(0u, 0u, 0u, 0u);
}

// Target offsets of the group members and row offsets of the tile.
template <int NT>
__device__ __forceinline__ void fill_offsets(const TcParams& p, uint64_t* toff, uint64_t* rowoff, int tid, int nthr) {
  for (int j = tid; j < (1 << NT); j += nthr) {
    uint64_t off = 0;
#pragma unroll
    for (int q = 0; q < NT; ++q)
      if ((j >> q) & 1) off |= 1ull << p.tpos[q];
    toff[j] = off;
  }
  for (int g = tid; g < kRows; g += nthr) {
    uint64_t off = 0;
    for (int b = 0, r = 0; b < p.tile_bits; ++b)
      if (!((p.tslot_mask >> b) & 1)) {
        if ((g >> r) & 1) off |= 1ull << p.P[b];
        ++r;
      }
    rowoff[g] = off;
  }
}

// column exponent field -> the increment it adds to a result's exponent field (K terms)
template <int K>
__host__ __device__ constexpr int column_scale(int field) {
  return (field - (1024 << 20)) - ((1022 + qsby::kScale + qsby::extra_bits(K)) << 20);   // in steps within 32 bits
}

// Row exponent fields [lim[0], lim[1]] whose results can have their exponent fields
// added (qsby::add_inc) in every column that is not all zeros.  The limits start at
// those of a column of exponent 0; limit_rows takes in a column's (csc: its largest
// high word, scale: its increment).
template <int K>
__device__ __forceinline__ void start_row_limits(int* lim) {
  constexpr int one = column_scale<K>(1023 << 20);
  lim[0] = qsby::kMinInc - one;
  lim[1] = qsby::kMaxInc - one;
}
__device__ __forceinline__ void limit_rows(int* lim, int csc, int scale) {
  if (csc == 0) return;
  atomicMax(lim, qsby::kMinInc - scale);
  atomicMin(lim + 1, qsby::kMaxInc - max(scale, qsby::kMaxInc - 0x7FFFFFFF));
}

// Per-CTA constants of a dense gate: the column scales and the digit slices of
// B, the initialising MMA's operands, the target offsets of the group members
// and the row offsets of the tile.
template <int NT, int NTHR>
__device__ void tile_constants(const TcParams& p, unsigned char* b_dig, unsigned char* a_pre, unsigned char* b_pre,
                               int* csc, int* lim, int* colsum, uint64_t* toff, uint64_t* rowoff, int tid) {
  constexpr int D = 1 << NT, K = 2 * D, N = 2 * D;
  if (tid == 0) start_row_limits<K>(lim);
  fill_start_rows(a_pre, tid, NTHR);
  fill_offsets<NT>(p, toff, rowoff, tid, NTHR);
  slice_matrix<NT, NTHR>(p, b_dig, N * K * 2, [](int n, int k) { return canon_off16(n, k, K); }, csc, colsum, tid);
  for (int idx = tid; idx < kLv * N; idx += NTHR) {
    const int L = idx / N, n = idx % N;
    fill_start_column(b_pre, L * N + n, qsby::start_value(L, K, colsum + n * kLv, qsby::extra_bits(K)));
  }
  for (int j = tid; j < D; j += NTHR) {
    const int mx = csc[2 * j], sc = column_scale<K>((int)qsby::row_field((uint32_t)mx));
    limit_rows(lim, mx, sc);
    csc[2 * j] = sc;
    csc[2 * j + 1] = sc;
  }
}

// Four outputs: levels -> Q -> double, scaled by the row's and the columns' powers of
// two.  rare: the row's exponent is beyond the limits.
template <int K>
__device__ __forceinline__ void finish_outputs(const float (*v)[4], int egs, const int* csc, bool rare, double* o) {
  const int4 s = *reinterpret_cast<const int4*>(csc);
  const int inc[4] = {egs + s.x, egs + s.y, egs + s.z, egs + s.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float u[kLv];
#pragma unroll
    for (int L = 0; L < kLv; ++L) u[L] = v[L][q];
    o[q] = __ll2double_rn(qsby::combine<K, qsby::extra_bits(K)>(u));
  }
  if (rare) {
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q] = qsby::mul_inc(o[q], inc[q]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q] = qsby::add_inc(o[q], inc[q]);
  }
}

// fp16 operand words of four amplitudes (hi, lo words of re and im) at the 16-byte
// column group `off` of every A slice
__device__ __forceinline__ void store_slices(unsigned char* A, uint32_t off, uint32_t abytes, const uint32_t (*R)[4],
                                             uint32_t ef1) {
  uint32_t pk[4][qsby::kA];
#pragma unroll
  for (int e = 0; e < 4; ++e)
    qsby::packed_digits(qsby::bytes_of(R[e][0], R[e][1], ef1), qsby::bytes_of(R[e][2], R[e][3], ef1), pk[e]);
#pragma unroll
  for (int s = 0; s < qsby::kA; ++s)
    *reinterpret_cast<uint4*>(A + s * abytes + off) = make_uint4(pk[0][s], pk[1][s], pk[2][s], pk[3][s]);
}

// two neighbouring amplitudes (32-byte aligned)
__device__ __forceinline__ void store_pair(void* at, const double* o) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(at), "d"(o[0]), "d"(o[1]), "d"(o[2]), "d"(o[3])
               : "memory");
}

// largest high word without sign of an amplitude's parts
__device__ __forceinline__ uint32_t max_abs(uint32_t m, const uint32_t* R) {
  return max(m, max(R[0] & 0x7FFFFFFFu, R[2] & 0x7FFFFFFFu));
}

}  // namespace

// ---------------------------------------------------------------------------
// Warp-specialised form for two to four targets (K <= 32, so every level
// starts at the magic and the epilogue reads level bit patterns directly).
// A unit is one tile, or two for three targets (as many amplitudes a unit as
// with four: one tile a unit, with four-deep rings, took 1.74 ms at 28 qubits
// against 1.50).  Eight producer warps gather units with cp.async into a ring of
// S staging slots (64 KB of loads in flight), take the row maxima (two threads
// per row, one shuffle) and write the digit slices into a ring of NA operand
// buffers; one thread issues the initialising MMA and the slice MMAs of each
// tile into a ring of NTM tensor-memory buffers; 16 epilogue warps (four per
// lane quarter, each a part of a row's columns) recombine, convert and store.
// Hand-offs are mbarriers: afull (producers -> MMA), aempty and accfull
// (MMA completion -> producers, epilogue), tempty (epilogue -> MMA) and
// mready (MMA thread -> epilogue, releasing onward the row exponents that the
// producers wrote into one of NM = NA + NTM metadata slots; a slot is
// rewritten only after the epilogue has finished the tile that used it).
// Every role steps its tile base by a masked add: with the inserted (target,
// row and control) bit positions filled with ones, adding the grid stride
// spread over the free positions carries through them.  Every wait is bounded
// and gives up when another role has.
// ---------------------------------------------------------------------------
namespace {
// epilogue and producer warps: with 8 and 8 the kernels waited for the epilogue
// (28 qubits, 3 / 4 targets 1.76 / 1.52 ms as eight warps of eight columns at a
// time, 1.91 / 1.65 of four; 16 warps 1.74 / 1.51)
constexpr int kWsE = 16, kWsP = 8;
constexpr int kWsThreads = 32 * (kWsE + kWsP + 1);  // and the MMA warp

__device__ __forceinline__ bool wait_ring(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  uint32_t spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    ++spins;
    if (spins > kWaitLimit || ((spins & 255u) == 0 && *abort_flag)) return true;
  }
  return false;
}

// the same for a whole warp: every lane gets the same answer, so a warp
// leaves its loop as one (its shuffles and tcgen05.ld need all lanes)
__device__ __forceinline__ bool wait_ring_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  return __any_sync(0xFFFFFFFFu, wait_ring(bar, parity, abort_flag)) != 0;
}

template <int NT>
struct Ws {
  static constexpr int D = 1 << NT, K = 2 * D, N = 2 * D;
  static constexpr int RB = NT == 3 ? 2 : 1;         // 128-row tiles that go through the rings as one unit
  static constexpr int LCOLS = kLv * N;              // accumulator columns of a tile
  static constexpr int NTM = 2;                      // accumulator buffers
  static constexpr int TSTRIDE = 512 / NTM;          // their column stride
  static constexpr int NA = 2;                       // operand buffers
  static constexpr int NM = NA + NTM;                // metadata slots
  static constexpr int S = 2;                        // staging slots (64 KB of loads in flight)
  static constexpr int PT = 32 * kWsP;               // producer threads
  static constexpr int EPP = D / 2;                  // amplitudes of a tile per producer thread (two per row)
  static constexpr int EPE = RB * D / (kWsE / 4);    // amplitudes of a unit per epilogue thread
  static constexpr int ABYTES = kRows * K * 2, BBYTES = N * K * 2;
  static constexpr int ABUF = RB * qsby::kA * ABYTES;   // operands of a unit
  static constexpr int SLOT = RB * PT * EPP * 16;
  static constexpr size_t a_off = 0;
  static constexpr size_t b_off = a_off + (size_t)NA * ABUF;
  static constexpr size_t apre_off = b_off + (size_t)qsby::kB * BBYTES;
  static constexpr size_t bpre_off = apre_off + kRows * 32;
  static constexpr size_t stg_off = bpre_off + (size_t)LCOLS * 32;
  static constexpr size_t toff_off = stg_off + (size_t)S * SLOT;
  static constexpr size_t rowoff_off = toff_off + 8 * D;
  static constexpr size_t bar_off = rowoff_off + 8 * kRows;
  static constexpr size_t csc_off = bar_off + 8 * (2 * NA + 2 * NTM + NM);
  static constexpr size_t ex_off = csc_off + 4 * N;
  static constexpr size_t colsum_off = ex_off + 4 * (size_t)NM * RB * kRows;
  static constexpr size_t slot_off = colsum_off + 4 * (size_t)kLv * N;
  static constexpr size_t lim_off = slot_off + 8;
  static constexpr size_t bytes = slot_off + 16;
  static_assert(RB * LCOLS <= TSTRIDE && NTM * TSTRIDE <= 512, "tensor memory");
  static_assert(bytes <= 227 * 1024, "shared memory");
  static_assert(K <= 32 && EPP % 4 == 0 && PT / kRows == 2, "mapping");
};

}  // namespace

template <int NT, bool PAIRS>
__global__ void __launch_bounds__(kWsThreads, 1) k_dense_ozaki_ws(double2* __restrict__ psi, const __grid_constant__ TcParams p) {
  using W = Ws<NT>;
  constexpr int K = W::K, N = W::N, NA = W::NA, NTM = W::NTM, NM = W::NM, S = W::S;
  constexpr int EPP = W::EPP, EPE = W::EPE, PT = W::PT, RB = W::RB;
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* a_dig = smem + W::a_off;
  unsigned char* b_dig = smem + W::b_off;
  unsigned char* a_pre = smem + W::apre_off;
  unsigned char* b_pre = smem + W::bpre_off;
  unsigned char* stg = smem + W::stg_off;
  uint64_t* toff = reinterpret_cast<uint64_t*>(smem + W::toff_off);
  uint64_t* rowoff = reinterpret_cast<uint64_t*>(smem + W::rowoff_off);
  uint64_t* afull = reinterpret_cast<uint64_t*>(smem + W::bar_off);
  uint64_t* aempty = afull + NA;
  uint64_t* accfull = aempty + NA;
  uint64_t* tempty = accfull + NTM;
  uint64_t* mready = tempty + NTM;
  int* csc = reinterpret_cast<int*>(smem + W::csc_off);
  int* meta_ex = reinterpret_cast<int*>(smem + W::ex_off);
  int* colsum = reinterpret_cast<int*>(smem + W::colsum_off);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + W::slot_off);
  int* lim = reinterpret_cast<int*>(smem + W::lim_off);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + W::slot_off + 4);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  tile_constants<NT, kWsThreads>(p, b_dig, a_pre, b_pre, csc, lim, colsum, toff, rowoff, tid);
  if (tid == 0) {
#pragma unroll
    for (int j = 0; j < NA; ++j) {
      mbar_init(afull + j, kWsP);        // one arrival per producer warp
      mbar_init(aempty + j, 1);
    }
#pragma unroll
    for (int k = 0; k < NTM; ++k) {
      mbar_init(accfull + k, 1);
      mbar_init(tempty + k, kWsE);       // one arrival per epilogue warp
    }
#pragma unroll
    for (int m = 0; m < NM; ++m) mbar_init(mready + m, 1);
    *abort_flag = 0;
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  fence_proxy_async();                        // B's slices and the initialising operands, for the MMAs
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  const int row_bits = p.tile_bits - NT;
  const uint64_t grid = gridDim.x, nunits = p.ntiles / RB;
  // unit u holds the tiles u RB + r, whose bases are x(u RB) | r rstep.
  // x(c) = insert_zeros(c); x(c + d) = ((x(c) | hole) + insert_zeros(d)) & ~hole
  uint64_t hole = 0;
  for (int q = 0; q < p.nhi; ++q) hole |= 1ull << p.hi_ins[q];
  const uint64_t gstep = insert_zeros(grid * RB, p.hi_ins, p.nhi);
  const uint64_t rstep = RB > 1 ? insert_zeros(1, p.hi_ins, p.nhi) : 0;
  auto step = [&](uint64_t x, uint64_t d) -> uint64_t { return ((x | hole) + d) & ~hole; };

  if (warp < kWsE) {
    // ---- epilogue: row g (tensor-memory lane) of tile r, amplitudes [l0, l0 + EPE) ----
    const int q = warp & 3;
    constexpr int PER = kWsE / 4 / RB;        // threads per row
    const int r = (warp >> 2) / PER, l0 = ((warp >> 2) % PER) * EPE;
    const int g = 32 * q + lane;
    const bool row_ok = g < (1 << row_bits);
    const uint32_t lane_addr = (uint32_t)(32 * q) << 16;
    uint64_t te[EPE];                         // byte offsets of this thread's amplitudes in a tile
#pragma unroll
    for (int i = 0; i < EPE; ++i) te[i] = (rowoff[g] | toff[l0 + i] | r * rstep) << 4;
    uint64_t xb = insert_zeros(blockIdx.x * (uint64_t)RB, p.hi_ins, p.nhi);
    for (int i = 0;; ++i, xb = step(xb, gstep)) {
      const uint64_t c = blockIdx.x + (uint64_t)i * grid;
      if (c >= nunits) break;
      const int k = i % NTM, m = i % NM;
      if (wait_ring_warp(mready + m, (uint32_t)(i / NM) & 1u, abort_flag)) {
        *abort_flag = 1;
        break;
      }
      const int egs = meta_ex[(m * RB + r) * kRows + g];
      const bool rare = egs < lim[0] || egs > lim[1];
      char* tp = reinterpret_cast<char*>(psi) + ((xb | p.ctrl_mask) << 4);
      if (wait_ring_warp(accfull + k, (uint32_t)(i / NTM) & 1u, abort_flag)) {
        *abort_flag = 1;
        break;
      }
      fence_after_sync();
      const uint32_t tb = tmem + (uint32_t)(k * W::TSTRIDE + r * W::LCOLS + 2 * l0) + lane_addr;
#pragma unroll
      for (int cc = 0; cc < 2 * EPE; cc += 4) {
        float v[kLv][4];
#pragma unroll
        for (int L = 0; L < kLv; ++L) tmem_ld4(tb + (uint32_t)(L * N + cc), v[L]);
        tmem_wait_ld();
        if (cc + 4 == 2 * EPE) {                // the buffer is read: hand it back to the MMA thread
          fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty + k);
        }
        if (row_ok) {
          double o[4];
          finish_outputs<K>(v, egs, csc + 2 * l0 + cc, rare, o);
          if (PAIRS) {
            store_pair(tp + te[cc >> 1], o);
          } else {
#pragma unroll
            for (int qq = 0; qq < 4; qq += 2)
              *reinterpret_cast<double2*>(tp + te[(cc + qq) >> 1]) = make_double2(o[qq], o[qq + 1]);
          }
        }
      }
    }
  } else if (warp < kWsE + kWsP) {
    // ---- producers: row g of every tile of the unit, part h (amplitudes [h EPP, (h + 1) EPP)) ----
    const int pt = tid - 32 * kWsE, pw = pt >> 5;
    // eight lanes (one 128-byte phase of a 16-byte store) hold eight rows of one
    // column group, so the slice stores meet no bank twice
    const int g = 16 * pw + (lane & 7) + 8 * (lane >> 4), h = (lane >> 3) & 1;
    const bool row_ok = g < (1 << row_bits);
    // Neighbours in pairs: lanes 2 i and 2 i + 1 copy each other's halves of a sector.
    // Copy i of a lane is amplitude (i & ~1) | (lane & 1) of the row of lane
    // (lane & ~1) | (i & 1), and goes to that thread's place: (i' PT + pt') 16 with
    // i' - i = pt - pt' = (lane & 1) - (i & 1).
    const int odd = lane & 1;
    const uint32_t swap[2] = {PAIRS ? (uint32_t)(odd * (PT - 1) * 16) : 0u, PAIRS ? (uint32_t)((odd - 1) * (PT - 1) * 16) : 0u};
    uint64_t tp[EPP];                         // byte offsets in a tile of the amplitudes that this thread copies
#pragma unroll
    for (int i = 0; i < EPP; ++i)
      tp[i] = PAIRS ? (rowoff[(g & ~1) | (i & 1)] | toff[h * EPP + ((i & ~1) | odd)]) << 4 : (rowoff[g] | toff[h * EPP + i]) << 4;
    const uint32_t stg_addr = smem_u32(stg) + (uint32_t)pt * 16u;
    auto issue = [&](uint64_t x, int slot) {
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const char* base = reinterpret_cast<const char*>(psi) + ((x | r * rstep | p.ctrl_mask) << 4);
#pragma unroll
        for (int i = 0; i < EPP; ++i)
          cp_async16(stg_addr + swap[i & 1] + (uint32_t)(slot * W::SLOT + (r * EPP + i) * PT * 16),
                     row_ok ? (const void*)(base + tp[i]) : psi, row_ok ? 16u : 0u);
      }
    };
    uint64_t xi = insert_zeros(blockIdx.x * (uint64_t)RB, p.hi_ins, p.nhi);   // base of the next tile to issue
#pragma unroll
    for (int sl = 0; sl < S; ++sl) {
      const uint64_t c = blockIdx.x + (uint64_t)sl * grid;
      if (c < nunits) issue(xi, sl);
      cp_async_commit();
      xi = step(xi, gstep);
    }
    for (int i = 0;; ++i) {
      const uint64_t c = blockIdx.x + (uint64_t)i * grid;
      if (c >= nunits) break;
      const int slot = i % S, j = i % NA, m = i % NM;
      cp_async_wait<S - 1>();
      if (PAIRS) __syncwarp();                // the other lane's copies, too
      uint32_t R[RB * EPP][4];
#pragma unroll
      for (int i2 = 0; i2 < RB * EPP; ++i2) {
        uint4 v;
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                     : "r"(stg_addr + (uint32_t)(slot * W::SLOT + i2 * PT * 16)));
        R[i2][0] = v.y;
        R[i2][1] = v.x;
        R[i2][2] = v.w;
        R[i2][3] = v.z;
      }
      // exponent fields of the rows (a row's other part is in lane xor 8)
      uint32_t em[RB];
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        em[r] = 0;
#pragma unroll
        for (int i2 = 0; i2 < EPP; ++i2) em[r] = max_abs(em[r], R[r * EPP + i2]);
        em[r] = qsby::row_field(max(em[r], __shfl_xor_sync(0xFFFFFFFFu, em[r], 8)));
      }
      // the slot's contents are in registers (used above): refill it S tiles ahead
      if (PAIRS) __syncwarp();
      {
        const uint64_t c2 = c + (uint64_t)S * grid;
        if (c2 < nunits) issue(xi, slot);
        cp_async_commit();
        xi = step(xi, gstep);
      }
      if (wait_ring_warp(aempty + j, ((uint32_t)(i / NA) & 1u) ^ 1u, abort_flag)) {
        *abort_flag = 1;
        break;
      }
      unsigned char* A = a_dig + j * W::ABUF;
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        if (h == 0) meta_ex[(m * RB + r) * kRows + g] = (int)em[r];
#pragma unroll
        for (int i2 = 0; i2 < EPP; i2 += 4)
          store_slices(A + r * qsby::kA * W::ABYTES, canon_off16(g, 2 * (h * EPP + i2), K), W::ABYTES, R + r * EPP + i2,
                       em[r] + 0x100000u);
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(afull + j);
    }
    cp_async_wait<0>();
  } else if (lane == 0) {
    // ---- MMA issue ----
    int last = -1;
    for (int i = 0;; ++i) {
      const uint64_t c = blockIdx.x + (uint64_t)i * grid;
      if (c >= nunits) break;
      const int j = i % NA, k = i % NTM, m = i % NM;
      if (wait_ring(afull + j, (uint32_t)(i / NA) & 1u, abort_flag)) {
        *abort_flag = 1;
        break;
      }
      mbar_arrive(mready + m);              // the producers' metadata, released onward to the epilogue
      if (wait_ring(tempty + k, ((uint32_t)(i / NTM) & 1u) ^ 1u, abort_flag)) {
        *abort_flag = 1;
        break;
      }
      fence_after_sync();
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const uint32_t dcol = tmem + (uint32_t)(k * W::TSTRIDE + r * W::LCOLS);
        mma_start<N>(dcol, a_pre, b_pre);
        mma_products<N, K / 16>(dcol, a_dig + j * W::ABUF + r * qsby::kA * W::ABYTES, b_dig);
      }
      mma_commit(aempty + j);
      mma_commit(accfull + k);
      last = i;
    }
    // the last tile's MMAs are complete before the tensor memory is freed
    if (last >= 0 && wait_ring(aempty + last % NA, (uint32_t)(last / NA) & 1u, abort_flag)) *abort_flag = 1;
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (tid == 0 && *abort_flag) atomicExch(p.err, 1);
  if (warp == 0) tmem_dealloc(tmem, 512);
}

template <int NT, bool PAIRS>
static cudaError_t dense_ozaki_ws(void* amps, const TcParams& p, cudaStream_t st) {
  constexpr size_t smem = Ws<NT>::bytes;
  static bool attr_done = false;
  if (!attr_done) {
    cudaError_t e = cudaFuncSetAttribute(k_dense_ozaki_ws<NT, PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  const uint64_t maxb = (uint64_t)num_sms(), nunits = p.ntiles / Ws<NT>::RB;
  if (nunits == 0) return cudaErrorInvalidValue;   // such passes go elsewhere (qs_api.cpp)
  const unsigned g = (unsigned)(nunits < maxb ? nunits : maxb);
  k_dense_ozaki_ws<NT, PAIRS><<<g, kWsThreads, smem, st>>>(static_cast<double2*>(amps), p);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Five targets (K = N = 64), in two blocks of 32 columns of K and of N, warp
// specialised.  16 producer warps (thread: row g, four amplitudes of each K
// block, in registers; a block's registers are reloaded for the next tile as
// soon as it is sliced) write one K block at a time into a ring of two operand
// buffers (56 KB each).  One thread issues the MMAs, N block 0 over both K
// blocks and then N block 1, into two accumulator buffers (256 columns each).
// Eight epilogue warps (two per lane quarter) recombine, convert and store one
// N block at a time.  B (64 KB) stays in shared memory.  So the MMAs on N block
// 0 of a tile run behind the epilogue of the previous tile's N block 1, those
// on N block 1 behind the epilogue of N block 0, and slicing behind both.
//
// Hand-offs are mbarriers: afull (producers -> MMA), aempty and accfull (MMA
// completion), tempty (epilogue -> MMA) and mready (MMA thread -> epilogue,
// releasing onward the row exponents that the producers wrote into one of four
// metadata slots; a slot is rewritten four tiles later, after the slicing of
// the tile before has waited for MMAs that waited for this tile's epilogue).
// Row maxima go through shared memory and one barrier of the producer warps per
// tile, which also carries the abort flag, so the producers leave together.
// Every wait is bounded and gives up at once when another role has.
// What bounds it: 10.3 thousand cycles per tile, of which the MMAs take 4.7 and
// neither the integer pipe (51%) nor issue (48%) is full; the operand buffers
// hold a single tile, so slicing the next one waits for the last MMAs on this
// one.  A third buffer does not fit in shared memory.  Twelve epilogue warps in
// place of eight (64 registers) took 2.53 ms against 2.30, and all phases in
// the same 16 warps 3.05.
// ---------------------------------------------------------------------------
namespace {
constexpr int kKnWarps = 16;                         // producer (five targets) or compute (six) warps
constexpr int kKnC = 32 * kKnWarps;
constexpr int kKnBlock = qsby::kB * 32 * 32 * 2;     // 16 KB: eight slices of a 32 x 32 block of B

// barrier of those warps; true for all if any thread says so
__device__ __forceinline__ bool compute_barrier_or(bool x) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n barrier.cta.red.or.pred p, 1, %2, q;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(r)
      : "r"((uint32_t)x), "n"(kKnC)
      : "memory");
  return r != 0;
}

// bounded wait that gives up at once when another role has, and says so
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return false;
  if (*abort_flag || wait_ring(bar, parity, abort_flag)) {
    *abort_flag = 1;
    return true;
  }
  return false;
}

// the same for a whole warp
__device__ __forceinline__ bool wait_or_abort_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  return __any_sync(0xFFFFFFFFu, wait_or_abort(bar, parity, abort_flag)) != 0;
}

// Epilogue of one N block (32 columns, accumulators at tb): a thread's row, NC of
// its columns from column c0 of the block on; csc0: their scales; rare: as for
// finish_outputs; addr(a): where amplitude a of those goes.  Hands the accumulators back on tempty once read.
template <int K, int NC, bool PAIRS, typename Addr>
__device__ __forceinline__ void epilogue_block(uint32_t tb, uint64_t* tempty, const int* csc0, int egs, bool rare,
                                               bool row_ok, int lane, const Addr& addr) {
#pragma unroll
  for (int cc = 0; cc < NC; cc += 4) {
    float v[kLv][4];
#pragma unroll
    for (int L = 0; L < kLv; ++L) tmem_ld4(tb + (uint32_t)(L * 32 + cc), v[L]);
    tmem_wait_ld();
    if (cc + 4 == NC) {
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty);
    }
    if (row_ok) {
      double o[4];
      finish_outputs<K>(v, egs, csc0 + cc, rare, o);
      if (PAIRS) {
        store_pair(addr(cc >> 1), o);
      } else {
#pragma unroll
        for (int q = 0; q < 4; q += 2) *addr((cc + q) >> 1) = make_double2(o[q], o[q + 1]);
      }
    }
  }
}

// Two neighbouring amplitudes at once.  With qubit 0 a target, an amplitude by itself
// uses half of a 32-byte sector, and its other half is read or written again by the
// thread's next access.
__device__ __forceinline__ void load_pair(const double2* at, double2* v) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(v[0].x), "=d"(v[0].y), "=d"(v[1].x), "=d"(v[1].y)
               : "l"(at)
               : "memory");
}

// the words of four amplitudes of a row (zeros beyond the last row); PAIRS: amplitudes
// 0, 1 and 2, 3 are neighbours in memory
template <bool PAIRS, typename Addr>
__device__ __forceinline__ void load_four(uint32_t (*R)[4], bool row_ok, const Addr& addr) {
#pragma unroll
  for (int i = 0; i < 4; i += 2) {
    double2 v[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    if (row_ok) {
      if (PAIRS) {
        load_pair(addr(i), v);
      } else {
        v[0] = *addr(i);
        v[1] = *addr(i + 1);
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      R[i + e][0] = (uint32_t)__double2hiint(v[e].x);
      R[i + e][1] = (uint32_t)__double2loint(v[e].x);
      R[i + e][2] = (uint32_t)__double2hiint(v[e].y);
      R[i + e][3] = (uint32_t)__double2loint(v[e].y);
    }
  }
}

// bits of the inserted (target, row and control) positions of a tile base
__device__ __forceinline__ uint64_t hole_mask(const TcParams& p) {
  uint64_t hole = 0;
  for (int q = 0; q < p.nhi; ++q) hole |= 1ull << p.hi_ins[q];
  return hole;
}

constexpr int kE5 = 8;                               // epilogue warps (two per lane quarter)
struct W5 {
  static constexpr int D = 32, K = 64, KB = 2, NM = 4;
  static constexpr int THREADS = 32 * (kE5 + kKnWarps + 1);
  static constexpr int ABYTES = kRows * 32 * 2, ABUF = qsby::kA * ABYTES;
  static constexpr size_t b_off = 2 * (size_t)ABUF;
  static constexpr size_t apre_off = b_off + (size_t)KB * KB * kKnBlock;
  static constexpr size_t bpre_off = apre_off + kRows * 32;
  static constexpr size_t toff_off = bpre_off + (size_t)KB * 8192;
  static constexpr size_t rowoff_off = toff_off + 8 * D;
  static constexpr size_t bar_off = rowoff_off + 8 * kRows;
  static constexpr size_t csc_off = bar_off + 8 * 14;
  static constexpr size_t max_off = csc_off + 4 * K;
  static constexpr size_t ex_off = max_off + 4 * 3 * kRows;
  static constexpr size_t colsum_off = ex_off + 4 * NM * kRows;
  static constexpr size_t slot_off = colsum_off + 4 * (size_t)kLv * K;
  static constexpr size_t lim_off = slot_off + 8;
  static constexpr size_t bytes = slot_off + 16;
  static_assert(bytes <= 227 * 1024, "shared memory");
};
}  // namespace

template <bool PAIRS>
__global__ void __launch_bounds__(W5::THREADS, 1)
    k_dense_ozaki5(double2* __restrict__ psi, const __grid_constant__ TcParams p) {
  using X = W5;
  constexpr int D = X::D, K = X::K, KB = X::KB;
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* a_dig = smem;
  unsigned char* b_dig = smem + X::b_off;
  unsigned char* a_pre = smem + X::apre_off;
  unsigned char* b_pre = smem + X::bpre_off;
  uint64_t* toff = reinterpret_cast<uint64_t*>(smem + X::toff_off);
  uint64_t* rowoff = reinterpret_cast<uint64_t*>(smem + X::rowoff_off);
  uint64_t* afull = reinterpret_cast<uint64_t*>(smem + X::bar_off);
  uint64_t *aempty = afull + 2, *accfull = afull + 4, *tempty = afull + 6, *mready = afull + 8, *done = afull + 12;
  int* csc = reinterpret_cast<int*>(smem + X::csc_off);
  int* rowmax = reinterpret_cast<int*>(smem + X::max_off);       // 3 x kRows
  int* meta_ex = reinterpret_cast<int*>(smem + X::ex_off);       // NM x kRows
  int* colsum = reinterpret_cast<int*>(smem + X::colsum_off);    // K x 8 (setup)
  int* lim = reinterpret_cast<int*>(smem + X::lim_off);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + X::slot_off);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + X::slot_off + 4);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  fill_start_rows(a_pre, tid, X::THREADS);
  fill_offsets<5>(p, toff, rowoff, tid, X::THREADS);
  if (tid == 0) start_row_limits<K>(lim);
  // B's slices in blocks of 32 x 32: block (K block, N block) at (kb KB + nb) 16 KB
  slice_matrix<5, X::THREADS>(
      p, b_dig, 2048,
      [](int n, int k) { return ((k >> 5) * KB + (n >> 5)) * kKnBlock + (int)canon_off16(n & 31, k & 31, 32); }, csc,
      colsum, tid);
  for (int idx = tid; idx < kLv * K; idx += X::THREADS) {
    const int L = idx / K, n = idx % K;
    fill_start_column(b_pre + (n >> 5) * 8192, L * 32 + (n & 31), qsby::start_value(L, K, colsum + n * kLv, qsby::extra_bits(K)));
  }
  for (int j = tid; j < D; j += X::THREADS) {
    const int mx = csc[2 * j], sc = column_scale<K>((int)qsby::row_field((uint32_t)mx));
    limit_rows(lim, mx, sc);
    csc[2 * j] = sc;
    csc[2 * j + 1] = sc;
  }
  for (int g = tid; g < 3 * kRows; g += X::THREADS) rowmax[g] = 0;
  if (tid == 0) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      mbar_init(afull + b, kKnWarps);        // one arrival per producer warp
      mbar_init(aempty + b, 1);
      mbar_init(accfull + b, 1);
      mbar_init(tempty + b, kE5);            // one arrival per epilogue warp
    }
#pragma unroll
    for (int m = 0; m < X::NM; ++m) mbar_init(mready + m, 1);
    mbar_init(done, 1);
    *abort_flag = 0;
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  fence_proxy_async();                        // B's slices and the initialising operands, for the MMAs
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  const uint64_t grid = gridDim.x;
  // tile bases: x(c) = insert_zeros(c); x(c + d) = ((x(c) | hole) + insert_zeros(d)) & ~hole
  const uint64_t hole = hole_mask(p), gstep = insert_zeros(grid, p.hi_ins, p.nhi);
  uint64_t xb = insert_zeros(blockIdx.x, p.hi_ins, p.nhi);

  if (warp < kE5) {
    // ---- epilogue: row g (tensor-memory lane), half h of each N block's columns ----
    const int g = 32 * (warp & 3) + lane, h = warp >> 2;
    const bool row_ok = g < (1 << (p.tile_bits - 5));
    const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
    const uint64_t roff = rowoff[g] | p.ctrl_mask;
    uint32_t it = 0;
    bool bad = false;
    for (uint64_t c = blockIdx.x; c < p.ntiles && !bad; c += grid, ++it, xb = ((xb | hole) + gstep) & ~hole) {
      const uint32_t m = it % X::NM;
      if (wait_or_abort_warp(mready + m, (it / X::NM) & 1u, abort_flag)) break;
      const int egs = meta_ex[m * kRows + g];
      const bool rare = egs < lim[0] || egs > lim[1];
      const uint64_t rb = xb | roff;
#pragma unroll
      for (int nb = 0; nb < 2; ++nb) {
        bad = wait_or_abort_warp(accfull + nb, it & 1u, abort_flag);
        if (bad) break;
        fence_after_sync();
        epilogue_block<K, 16, PAIRS>(tmem + (uint32_t)(256 * nb + 16 * h) + lane_addr, tempty + nb, csc + 32 * nb + 16 * h, egs,
                              rare, row_ok, lane, [&](int a) { return psi + (rb | toff[16 * nb + 8 * h + a]); });
      }
    }
  } else if (warp < kE5 + kKnWarps) {
    // ---- producers: row g, amplitudes 16 kb + 4 cg + i (i < 4) of each K block ----
    const int pw = warp - kE5, g = 32 * (pw & 3) + lane, cg = pw >> 2;
    const bool row_ok = g < (1 << (p.tile_bits - 5));
    const uint64_t roff = rowoff[g] | p.ctrl_mask;
    const uint32_t a_addr = canon_off16(g, 8 * cg, 32);
    uint32_t R[KB * 4][4];
    uint64_t rb = xb | roff;
#pragma unroll
    for (int kb = 0; kb < KB; ++kb)
      load_four<PAIRS>(R + 4 * kb, row_ok, [&](int i) { return psi + (rb | toff[16 * kb + 4 * cg + i]); });
    uint32_t it = 0;
    bool bad = false;
    for (uint64_t c = blockIdx.x; c < p.ntiles; c += grid, ++it) {
      const uint32_t slot = it % 3;
      uint32_t mx = 0;
#pragma unroll
      for (int i = 0; i < KB * 4; ++i) mx = max_abs(mx, R[i]);
      atomicMax(rowmax + slot * kRows + g, (int)mx);   // the four threads of a row are in different warps
      if (compute_barrier_or(bad || *abort_flag)) break;
      const uint32_t ef = qsby::row_field((uint32_t)rowmax[slot * kRows + g]);   // exponent field of the row
      if (cg == 0) {
        // the previous tile's slot: read by every warp before this barrier, next
        // written after the following one
        rowmax[(slot == 0 ? 2 : slot - 1) * kRows + g] = 0;
        meta_ex[(it % X::NM) * kRows + g] = (int)ef;
      }
      const bool has_next = c + grid < p.ntiles;
      xb = ((xb | hole) + gstep) & ~hole;
      rb = xb | roff;
#pragma unroll
      for (int kb = 0; kb < KB; ++kb) {
        if (it > 0) bad |= wait_or_abort_warp(aempty + kb, (it - 1) & 1u, abort_flag);
        store_slices(a_dig + kb * X::ABUF, a_addr, X::ABYTES, R + 4 * kb, ef + 0x100000u);
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(afull + kb);
        if (has_next) load_four<PAIRS>(R + 4 * kb, row_ok, [&](int i) { return psi + (rb | toff[16 * kb + 4 * cg + i]); });
      }
    }
  } else if (lane == 0) {
    // ---- MMA issue ----
    uint32_t it = 0;
    bool bad = false;
    for (uint64_t c = blockIdx.x; c < p.ntiles && !bad; c += grid, ++it) {
      for (int nb = 0; nb < 2 && !bad; ++nb) {
        if (it > 0) bad = wait_or_abort(tempty + nb, (it - 1) & 1u, abort_flag);
        if (bad) break;
        fence_after_sync();
        const uint32_t dcol = tmem + 256u * nb;
        mma_start<32>(dcol, a_pre, b_pre + nb * 8192);
        for (int kb = 0; kb < KB && !bad; ++kb) {
          if (nb == 0) {
            bad = wait_or_abort(afull + kb, it & 1u, abort_flag);
            fence_after_sync();
            if (kb == KB - 1) mbar_arrive(mready + it % X::NM);   // the producers' metadata, released onward
          }
          if (!bad) mma_products<32, 2>(dcol, a_dig + kb * X::ABUF, b_dig + (kb * KB + nb) * kKnBlock);
          if (nb == 1) mma_commit(aempty + kb);
        }
        mma_commit(accfull + nb);
      }
    }
    // every MMA is complete before the tensor memory is freed
    mma_commit(done);
    if (wait_phase(done, 0)) *abort_flag = 1;
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (tid == 0 && *abort_flag) atomicExch(p.err, 1);
  if (warp == 0) tmem_dealloc(tmem, 512);
}

template <bool PAIRS>
static cudaError_t dense_ozaki5(void* amps, const TcParams& p, cudaStream_t st) {
  static bool attr_done = false;
  if (!attr_done) {
    cudaError_t e = cudaFuncSetAttribute(k_dense_ozaki5<PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W5::bytes);
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  const uint64_t maxb = (uint64_t)num_sms();
  const unsigned g = (unsigned)(p.ntiles < maxb ? p.ntiles : maxb);
  k_dense_ozaki5<PAIRS><<<g, W5::THREADS, W5::bytes, st>>>(static_cast<double2*>(amps), p);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Six targets (K = N = 128), in four blocks of 32 columns of K and of N.  16
// compute warps hold a tile's amplitudes in registers (thread: row g, four
// amplitudes of each K block), slice one K block at a time into a ring of two
// operand buffers, and recombine one N block at a time out of two accumulator
// buffers.  Reading all inputs into registers first makes the update in place
// safe.  One thread issues the MMAs: for a pair of N blocks, every K block
// against both.  The second pair takes the K blocks in the order 3, 2, 1, 0, so
// that two of its four are still in the operand buffers.  B's slices (256 KB)
// do not fit in shared memory: a setup kernel (k_wide_matrix) writes them to the
// caller's scratch, and another warp streams the 16 KB block of each (K, N) pair
// from L2 into a ring of four slots with bulk copies.  Hand-offs as for five
// targets, with bfull (bulk copy) and bempty (MMA completion) for B's slots.
// Rows that the slices cannot hold as FP64 did (an infinity or NaN, amplitudes all below
// 2^-965, results near the ends of the exponent range) are left alone and then made in
// FP64, one warp a row.
// Bound by the tensor cores (53% busy, two fifths of each tile's time being the
// epilogues and slicing that share its 16 warps): 34.7 thousand cycles per tile.
// ---------------------------------------------------------------------------
namespace {
// layout of the scratch that k_wide_matrix fills
constexpr int kWideStart = 16 * kKnBlock;            // four start operands (N block) of 256 columns x 32 bytes
constexpr int kWideScale = kWideStart + 4 * 8192;    // of 128 columns: exponent increment, largest high word
constexpr int kWideFlag = kWideScale + 8 * 128;      // kWideFlags flags: the matrix does not mix the group
static_assert(kWideFlag + 4 * kWideFlags <= (int)kWideScratch && kWideFlags == 128, "scratch of the six-target kernel");
// An output whose coefficients all lie within 2^-kMixBits of the largest depends on
// every amplitude of its group, the largest among them.
constexpr uint32_t kMixBits = 16;

struct W6 {
  static constexpr int D = 64, K = 128, KB = 4;
  static constexpr int THREADS = kKnC + 64;
  static constexpr int ABYTES = kRows * 32 * 2, ABUF = qsby::kA * ABYTES;
  static constexpr size_t b_off = 2 * (size_t)ABUF;
  static constexpr size_t apre_off = b_off + 4 * (size_t)kKnBlock;
  static constexpr size_t bpre_off = apre_off + kRows * 32;
  static constexpr size_t toff_off = bpre_off + (size_t)KB * 8192;
  static constexpr size_t rowoff_off = toff_off + 8 * D;
  static constexpr size_t bar_off = rowoff_off + 8 * kRows;
  static constexpr size_t csc_off = bar_off + 8 * 18;
  static constexpr size_t max_off = csc_off + 4 * K;
  static constexpr size_t slot_off = max_off + 4 * 3 * kRows;
  static constexpr size_t lim_off = slot_off + 8;
  static constexpr size_t bytes = slot_off + 16;
  static_assert(bytes <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// K block of step j of pass np over K: the second pass goes back
__device__ __forceinline__ int k_block(int np, int j) { return np ? W6::KB - 1 - j : j; }

// One group (amplitudes at base | target bits) in FP64 by one warp, with the sums of the
// FP64 kernel: a lane holds two amplitudes and two outputs.
__device__ __noinline__ void group_f64(double2* psi, uint64_t base, const TcParams& p, int lane) {
  uint64_t at[2] = {base, base};
#pragma unroll
  for (int e = 0; e < 2; ++e)
    for (int q = 0; q < 6; ++q)
      if ((lane + 32 * e) >> p.mbit[q] & 1) at[e] |= 1ull << p.tpos[q];
  const double2 x[2] = {psi[at[0]], psi[at[1]]};
  const double2* m = reinterpret_cast<const double2*>(p.mat) + 64 * lane;
  double2 y[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
  for (int l = 0; l < 64; ++l) {
    const double xr = __shfl_sync(0xFFFFFFFFu, l < 32 ? x[0].x : x[1].x, l & 31);
    const double xi = __shfl_sync(0xFFFFFFFFu, l < 32 ? x[0].y : x[1].y, l & 31);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      double2 c = m[2048 * e + l];
      if (p.conj) c.y = -c.y;
      y[e].x = fma(c.x, xr, y[e].x);
      y[e].x = fma(-c.y, xi, y[e].x);
      y[e].y = fma(c.x, xi, y[e].y);
      y[e].y = fma(c.y, xr, y[e].y);
    }
  }
  psi[at[0]] = y[0];
  psi[at[1]] = y[1];
}
}  // namespace

// One block per column of the realified six-target matrix, one thread per row:
// digits into the 32 x 32 blocks of the scratch, start operands, column scale.
//
// Also whether the byte slices may stand in for FP64.  They hold an amplitude to 2^-55
// of the largest of its group.  Where every output depends on that largest one that is
// what an output can be held to (rounding errors of FP64 sums are of its size too), but
// a matrix with zeros (a permutation, a diagonal, a gate with controls of its own) keeps
// small amplitudes apart from large ones, and FP64 then keeps all their bits.  So a
// matrix with an entry below 2^-16 of its row's largest, or one that is not finite, raises
// a flag: k_dense_ozaki6 returns, and the FP64 kernel (or the double-float one, by the
// handle's arithmetic) that is launched after it, and returns otherwise, makes the
// pass.  2^-16: of Haar matrices one in 200 thousand has such an entry.  28 qubits,
// spread targets: 3.96 ms mixing, 111 ms in FP64; the kernel that returns takes 2 us and
// a launch (calls at 2^7 to 2^18 amplitudes 38 to 42 us without it, 43 to 47 with it).
__global__ void __launch_bounds__(128) k_wide_matrix(const __grid_constant__ TcParams p, unsigned char* __restrict__ out) {
  constexpr int D = 64, K = 128;
  __shared__ int mx, sums[kLv];
  const int n = blockIdx.x, k = threadIdx.x;
  if (k < kLv) sums[k] = 0;
  if (k == 0) mx = 0;
  __syncthreads();
  const double2 m = matrix_entry(p, D, n >> 1, k >> 1);
  const double v = (n & 1) ? ((k & 1) ? m.x : m.y) : ((k & 1) ? -m.y : m.x);
  atomicMax(&mx, __double2hiint(v) & 0x7FFFFFFF);
  __syncthreads();
  const bool flag = __syncthreads_or(mx >= 0x7FF00000 || max(abs_hi(m.x), abs_hi(m.y)) + (kMixBits << 20) < (uint32_t)mx);
  const uint32_t ef = qsby::row_field((uint32_t)mx);
  int d[qsby::kB];
  qsby::digits_b((uint32_t)__double2hiint(v), (uint32_t)__double2loint(v), ef, d);
  unsigned char* blk = out + ((k >> 5) * 4 + (n >> 5)) * kKnBlock + canon_off16(n & 31, k & 31, 32);
#pragma unroll
  for (int t = 0; t < qsby::kB; ++t) {
    *reinterpret_cast<uint16_t*>(blk + t * 2048) = half_bits(d[t]);
    atomicAdd(sums + t, d[t]);
  }
  __syncthreads();
  if (k < kLv)
    fill_start_column(out + kWideStart + (n >> 5) * 8192, k * 32 + (n & 31), qsby::start_value(k, K, sums, qsby::extra_bits(K)));
  if (k == 0) {
    int* col = reinterpret_cast<int*>(out + kWideScale) + 2 * n;
    col[0] = column_scale<K>((int)ef);
    col[1] = mx;
    reinterpret_cast<int*>(out + kWideFlag)[n] = flag;
  }
}

template <bool PAIRS>
__global__ void __launch_bounds__(W6::THREADS, 1)
    k_dense_ozaki6(double2* __restrict__ psi, const __grid_constant__ TcParams p, const unsigned char* __restrict__ wide) {
  using X = W6;
  if (any_flag(reinterpret_cast<const int*>(wide + kWideFlag))) return;
  constexpr int K = X::K, KB = X::KB, NPASS = 2;
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* a_dig = smem;
  unsigned char* b_dig = smem + X::b_off;
  unsigned char* a_pre = smem + X::apre_off;
  unsigned char* b_pre = smem + X::bpre_off;
  uint64_t* toff = reinterpret_cast<uint64_t*>(smem + X::toff_off);
  uint64_t* rowoff = reinterpret_cast<uint64_t*>(smem + X::rowoff_off);
  uint64_t* afull = reinterpret_cast<uint64_t*>(smem + X::bar_off);
  uint64_t *aempty = afull + 2, *accfull = afull + 4, *tempty = afull + 6, *bfull = afull + 8, *bempty = afull + 12,
           *done = afull + 16;
  int* csc = reinterpret_cast<int*>(smem + X::csc_off);
  int* rowmax = reinterpret_cast<int*>(smem + X::max_off);       // 3 x kRows
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + X::slot_off);
  int* lim = reinterpret_cast<int*>(smem + X::lim_off);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + X::slot_off + 4);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint4* src = reinterpret_cast<const uint4*>(wide + kWideStart);
  for (int i = tid; i < KB * 8192 / 16; i += X::THREADS) reinterpret_cast<uint4*>(b_pre)[i] = src[i];
  if (tid == 0) start_row_limits<K>(lim);
  __syncthreads();
  for (int n = tid; n < K; n += X::THREADS) {
    const int* col = reinterpret_cast<const int*>(wide + kWideScale) + 2 * n;
    limit_rows(lim, col[1], col[0]);
    csc[n] = col[0];
  }
  fill_start_rows(a_pre, tid, X::THREADS);
  fill_offsets<6>(p, toff, rowoff, tid, X::THREADS);
  for (int g = tid; g < 3 * kRows; g += X::THREADS) rowmax[g] = 0;
  if (tid == 0) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      mbar_init(afull + b, kKnWarps);        // one arrival per compute warp
      mbar_init(aempty + b, 1);
      mbar_init(accfull + b, 1);
      mbar_init(tempty + b, kKnWarps);
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      mbar_init(bfull + b, 1);
      mbar_init(bempty + b, 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  fence_proxy_async();                        // the initialising operands, for the MMAs
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  const uint64_t grid = gridDim.x;
  // tile bases: x(c) = insert_zeros(c); x(c + d) = ((x(c) | hole) + insert_zeros(d)) & ~hole
  const uint64_t hole = hole_mask(p), gstep = insert_zeros(grid, p.hi_ins, p.nhi);

  if (warp < kKnWarps) {
    const int g = 32 * (warp & 3) + lane, cg = warp >> 2;         // row (tensor-memory lane), column group
    const bool row_ok = g < (1 << (p.tile_bits - 6));
    const uint64_t roff = rowoff[g] | p.ctrl_mask;
    const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
    const uint32_t a_addr = canon_off16(g, 8 * cg, 32);
    uint32_t R[KB * 4][4];                    // amplitudes 16 kb + 4 cg + i of the row, i < 4
    uint32_t fills[2] = {0, 0}, reads[2] = {0, 0};   // uses of the operand and accumulator buffers so far
    bool bad = false;
    uint64_t xb = insert_zeros(blockIdx.x, p.hi_ins, p.nhi);
    uint64_t rb = xb | roff;
#pragma unroll
    for (int kb = 0; kb < KB; ++kb)
      load_four<PAIRS>(R + 4 * kb, row_ok, [&](int i) { return psi + (rb | toff[16 * kb + 4 * cg + i]); });
    uint32_t it = 0;
    for (uint64_t c = blockIdx.x; c < p.ntiles; c += grid, ++it) {
      const uint32_t slot = it % 3;
      uint32_t mx = 0;
#pragma unroll
      for (int i = 0; i < KB * 4; ++i) mx = max_abs(mx, R[i]);
      atomicMax(rowmax + slot * kRows + g, (int)mx);   // the four threads of a row are in different warps
      if (compute_barrier_or(bad || *abort_flag)) break;
      const uint32_t mr = (uint32_t)rowmax[slot * kRows + g];
      const uint32_t ef = qsby::row_field(mr);   // exponent field of the row
      // the previous tile's slot: read by every warp before this barrier, next
      // written after the following one
      if (cg == 0) rowmax[(slot == 0 ? 2 : slot - 1) * kRows + g] = 0;
      // a row that is not finite, below the slices' range, or whose results may be: its
      // amplitudes stay as they are until the tile is done
      const bool far = row_ok && mr != 0 && (mr >= 0x7FF00000u || mr < (uint32_t)qsby::kFloor << 20 ||
                                             (int)ef < lim[0] || (int)ef > lim[1]);
      const bool has_next = c + grid < p.ntiles;
      xb = ((xb | hole) + gstep) & ~hole;
      const uint64_t rb_next = xb | roff;
#pragma unroll
      for (int np = 0; np < NPASS; ++np) {
#pragma unroll
        for (int j = 0; j < KB; ++j) {
          if (np > 0 && j < 2) continue;      // still in the operand buffers
          const int kb = k_block(np, j), b = kb & 1;
          if (fills[b] > 0) bad |= wait_or_abort_warp(aempty + b, (fills[b] - 1) & 1u, abort_flag);
          ++fills[b];
          store_slices(a_dig + b * X::ABUF, a_addr, X::ABYTES, R + 4 * kb, ef + 0x100000u);
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(afull + b);
          // the last use of these registers in this tile
          if (has_next && (np > 0 || kb >= 2))
            load_four<PAIRS>(R + 4 * kb, row_ok, [&](int i) { return psi + (rb_next | toff[16 * kb + 4 * cg + i]); });
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int nb = 2 * np + h;
          bad |= wait_or_abort_warp(accfull + h, reads[h] & 1u, abort_flag);
          ++reads[h];
          fence_after_sync();
          epilogue_block<K, 8, PAIRS>(tmem + (uint32_t)(256 * h + 8 * cg) + lane_addr, tempty + h, csc + 32 * nb + 8 * cg, (int)ef,
                               false, row_ok && !far, lane, [&](int a) { return psi + (rb | toff[16 * nb + 4 * cg + a]); });
        }
      }
      if (cg == 0)
        for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, far); todo != 0; todo &= todo - 1)
          group_f64(psi, __shfl_sync(0xFFFFFFFFu, rb, __ffs(todo) - 1), p, lane);
      rb = rb_next;
    }
  } else if (warp == kKnWarps && lane == 0) {
    // ---- MMA issue ----
    uint32_t fills[2] = {0, 0}, writes[2] = {0, 0}, nblk = 0;
    bool bad = false;
    for (uint64_t c = blockIdx.x; c < p.ntiles && !bad; c += grid)
      for (int np = 0; np < NPASS && !bad; ++np)
        for (int j = 0; j < KB && !bad; ++j) {
          const int kb = k_block(np, j), b = kb & 1;
          if (np == 0 || j >= 2) {
            bad = wait_or_abort(afull + b, fills[b] & 1u, abort_flag);
            ++fills[b];
          }
          for (int h = 0; h < 2 && !bad; ++h) {
            const uint32_t dcol = tmem + 256u * h;
            if (j == 0) {
              if (writes[h] > 0) bad = wait_or_abort(tempty + h, (writes[h] - 1) & 1u, abort_flag);
              ++writes[h];
            }
            const uint32_t slot = nblk & 3u;
            if (!bad) bad = wait_or_abort(bfull + slot, (nblk >> 2) & 1u, abort_flag);
            if (bad) break;
            ++nblk;
            fence_after_sync();
            if (j == 0) mma_start<32>(dcol, a_pre, b_pre + (2 * np + h) * 8192);
            mma_products<32, 2>(dcol, a_dig + b * X::ABUF, b_dig + slot * kKnBlock);
            mma_commit(bempty + slot);
            if (j == KB - 1) mma_commit(accfull + h);
          }
          // the buffer is free unless the next pass starts with it
          if (np > 0 || j < 2) mma_commit(aempty + b);
        }
    // every MMA is complete before the tensor memory is freed
    mma_commit(done);
    if (wait_phase(done, 0)) *abort_flag = 1;
  } else if (warp == kKnWarps + 1 && lane == 0) {
    // ---- B blocks, in the order of the MMA thread ----
    uint32_t nblk = 0;
    bool bad = false;
    for (uint64_t c = blockIdx.x; c < p.ntiles && !bad; c += grid)
      for (int np = 0; np < NPASS && !bad; ++np)
        for (int j = 0; j < KB && !bad; ++j)
          for (int h = 0; h < 2; ++h, ++nblk) {
            const uint32_t slot = nblk & 3u;
            if (nblk >= 4) bad = wait_or_abort(bempty + slot, ((nblk >> 2) - 1) & 1u, abort_flag);
            if (bad) break;
            bulk_load(smem_u32(b_dig) + slot * kKnBlock, wide + (k_block(np, j) * KB + 2 * np + h) * kKnBlock, kKnBlock,
                      bfull + slot);
          }
    // every copy has arrived before the CTA ends (the last fill of each slot)
    for (uint32_t s = 0; s < 4; ++s) {
      const uint32_t f = nblk > s ? (nblk - s + 3) / 4 : 0;       // fills of slot s
      if (f > 0 && wait_phase(bfull + s, (f - 1) & 1u)) *abort_flag = 1;
    }
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  if (tid == 0 && *abort_flag) atomicExch(p.err, 1);
  if (warp == 0) tmem_dealloc(tmem, 512);
}

template <bool PAIRS>
static cudaError_t dense_ozaki6(void* amps, const TcParams& p, void* scratch, cudaStream_t st) {
  static bool attr_done = false;
  if (!attr_done) {
    cudaError_t e = cudaFuncSetAttribute(k_dense_ozaki6<PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W6::bytes);
    // the three kernels of a pass in one split of shared memory and L1 (changing it
    // between them took 3 us a call)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_wide_matrix, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  unsigned char* wide = static_cast<unsigned char*>(scratch);
  k_wide_matrix<<<W6::K, W6::K, 0, st>>>(p, wide);
  const uint64_t maxb = (uint64_t)num_sms();
  const unsigned g = (unsigned)(p.ntiles < maxb ? p.ntiles : maxb);
  k_dense_ozaki6<PAIRS><<<g, W6::THREADS, W6::bytes, st>>>(static_cast<double2*>(amps), p, wide);
  return cudaGetLastError();
}

template <bool PAIRS>
static cudaError_t dense_ozaki(void* amps, const TcParams& p, void* scratch, cudaStream_t st) {
  switch (p.n) {
    case 3: return dense_ozaki_ws<3, PAIRS>(amps, p, st);
    case 4: return dense_ozaki_ws<4, PAIRS>(amps, p, st);
    case 5: return dense_ozaki5<PAIRS>(amps, p, st);
    case 6: return dense_ozaki6<PAIRS>(amps, p, scratch, st);
    default: return cudaErrorInvalidValue;
  }
}

// With qubit 0 a target, amplitudes 2 i and 2 i + 1 of a row are neighbours in memory:
// they move together (32 bytes, a whole sector).  28 qubits, ms, one by one / in
// pairs: 3, 4, 5, 6 targets on qubits 0, 1, ...: 2.50 / 2.27, 3.01 / 2.34, 3.32 / 2.73, 5.03 / 4.33; on
// qubit 0 and high ones: 1.94 / 1.71, 1.99 / 1.77, 2.25 / 2.20, 3.92 / 3.86.  Other
// passes keep the plain form: the exchange costs the producers up to 8% there.
cudaError_t launch_dense_ozaki(void* amps, const TcParams& p, void* scratch, cudaStream_t st, const int** when) {
  if (when) *when = p.n == 6 ? reinterpret_cast<const int*>(static_cast<unsigned char*>(scratch) + kWideFlag) : nullptr;
  if (p.tpos[0] == 0 && p.tile_bits > p.n) return dense_ozaki<true>(amps, p, scratch, st);
  return dense_ozaki<false>(amps, p, scratch, st);
}

}  // namespace qsk
