// Tile passes of planned complex64 circuits (qs_tile.h): one block per tile reads
// 2^12 amplitudes into shared memory, runs the pass's sweeps and writes them back.
//
// What bounds it: instruction issue (about two thirds of the slots), then the FP32
// pipe; a pass by itself costs one read and one write of the state (1.27 ms at 29
// qubits), and for 16 amplitudes a sweep adds 16 shared loads, 16 stores and some 50
// index instructions a thread, a one-target gate 64 packed multiply-adds and 32 moves,
// a two-target gate 128 and 32, a gadget 64 (32 with an odd number of Y) and 15 for
// signs.  150 random gates at 29 qubits, 17 passes: 44 ms, 48 with one operation an
// instruction, against 94 in dense blocks of at most six qubits.
// Four 256-thread blocks a multiprocessor (64 registers a thread): one block's
// sweeps run while the others' loads and stores are in flight (tiles of 2^13 with
// two 512-thread blocks, 15 passes: 49.7 against 48.0 ms).  Matrices come from shared
// memory: indexed reads of the constant bank took 82 ms.
#include "qs_device.cuh"
#include "qs_internal.h"
#include "qs_tile.h"

namespace qsk {
namespace {

using namespace qstile;

constexpr int kTileThreads = 1 << kThreadBits;
constexpr size_t kTileSmem = (sizeof(float2) << kPassBits) + sizeof(float) * kMaxCoef;

// Two FP32 operations at once on a (re, im) pair.
__device__ __forceinline__ unsigned long long& bits(float2& v) { return reinterpret_cast<unsigned long long&>(v); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(bits(d)) : "l"(bits(a)), "l"(bits(b)));
  return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(bits(d)) : "l"(bits(a)), "l"(bits(b)), "l"(bits(c)));
  return d;
}

// Entry e of a matrix at shared address u: (re, re) and (-im, im).  Volatile:
// loaded where it is used, so that a matrix is not kept in registers beside the 32 of
// the amplitudes.
struct Entry {
  float2 r, i;
};
__device__ __forceinline__ Entry entry(uint32_t u, int e) {
  Entry m;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(bits(m.r)), "=l"(bits(m.i)) : "r"(u + 16 * e));
  return m;
}

// ok: bit r = the controls are set at register r (C; otherwise they are everywhere)
template <int K, bool C>
__device__ __forceinline__ void gate1(float2 (&a)[kSweepAmps], uint32_t u, uint32_t ok) {
  const Entry m0 = entry(u, 0), m1 = entry(u, 1), m2 = entry(u, 2), m3 = entry(u, 3);
#pragma unroll
  for (int r = 0; r < kSweepAmps; ++r) {
    if (r >> K & 1) continue;
    if (C && !(ok >> r & 1u)) continue;
    const float2 x = a[r], y = a[r | 1 << K], xs = make_float2(x.y, x.x), ys = make_float2(y.y, y.x);
    a[r] = fma2(m1.i, ys, fma2(m1.r, y, fma2(m0.i, xs, mul2(m0.r, x))));
    a[r | 1 << K] = fma2(m3.i, ys, fma2(m3.r, y, fma2(m2.i, xs, mul2(m2.r, x))));
  }
}

template <int K0, int K1, bool C>
__device__ __forceinline__ void gate2(float2 (&a)[kSweepAmps], uint32_t u, uint32_t ok) {
#pragma unroll
  for (int r = 0; r < kSweepAmps; ++r) {
    if ((r >> K0 & 1) || (r >> K1 & 1)) continue;
    if (C && !(ok >> r & 1u)) continue;
    float2 o[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const float2 v = a[r | (l & 1) << K0 | (l >> 1) << K1], vs = make_float2(v.y, v.x);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const Entry m = entry(u, 4 * j + l);
        o[j] = l == 0 ? mul2(m.r, v) : fma2(m.r, v, o[j]);
        o[j] = fma2(m.i, vs, o[j]);
      }
    }
#pragma unroll
    for (int l = 0; l < 4; ++l) a[r | (l & 1) << K0 | (l >> 1) << K1] = o[l];
  }
}

template <bool C>
__device__ __forceinline__ void dense(float2 (&a)[kSweepAmps], const TileOp& op, uint32_t u, uint32_t ok) {
  if (op.kind == OP_GATE1) {
    if (op.k == 0) gate1<0, C>(a, u, ok);
    if (op.k == 1) gate1<1, C>(a, u, ok);
    if (op.k == 2) gate1<2, C>(a, u, ok);
    if (op.k == 3) gate1<3, C>(a, u, ok);
  } else {
    if (op.k == 0) gate2<0, 1, C>(a, u, ok);
    if (op.k == 1) gate2<0, 2, C>(a, u, ok);
    if (op.k == 2) gate2<0, 3, C>(a, u, ok);
    if (op.k == 3) gate2<1, 2, C>(a, u, ok);
    if (op.k == 4) gate2<1, 3, C>(a, u, ok);
    if (op.k == 5) gate2<2, 3, C>(a, u, ok);
  }
}

// a_r <- c a_r + s_r i^IM a_{r ^ M}; s_r = s with its sign changed by the parity of
// r & y (the sign of register 0 is in s already)
template <int M, bool IM>
__device__ __forceinline__ void gadget(float2 (&a)[kSweepAmps], float c, uint32_t s, uint32_t y) {
  uint32_t t[kSweepAmps];
  t[0] = s;
#pragma unroll
  for (int r = 1; r < kSweepAmps; ++r) {
    const int low = r & -r, b = low == 1 ? 0 : low == 2 ? 1 : low == 4 ? 2 : 3;
    t[r] = t[r ^ low] ^ (y >> b & 1u) << 31;
  }
#pragma unroll
  for (int r = 0; r < kSweepAmps; ++r) {
    const int q = r ^ M;
    if (q < r) continue;
    const float sr = __uint_as_float(t[r]), sq = __uint_as_float(t[q]);
    const float2 x = a[r], z = a[q];
    if (IM) {
      a[r] = make_float2(c * x.x - sr * z.y, c * x.y + sr * z.x);
      if (q != r) a[q] = make_float2(c * z.x - sq * x.y, c * z.y + sq * x.x);
    } else {
      const float2 cc = make_float2(c, c);
      a[r] = fma2(make_float2(sr, sr), z, mul2(cc, x));
      if (q != r) a[q] = fma2(make_float2(sq, sq), x, mul2(cc, z));
    }
  }
}

// (Separate ifs, not a switch: joins of two paths keep the amplitudes in their
// registers, a join of many made the compiler spill 900 bytes.)
template <int M>
__device__ __forceinline__ void gadget_m(float2 (&a)[kSweepAmps], uint32_t k, float c, uint32_t s, uint32_t y) {
  if (k == M) gadget<M, false>(a, c, s, y);
  if (k == (M | 16)) gadget<M, true>(a, c, s, y);
}

template <int M>
__device__ __forceinline__ void gadget_4m(float2 (&a)[kSweepAmps], uint32_t k, float c, uint32_t s, uint32_t y) {
  if ((k & 12) != M) return;
  gadget_m<M>(a, k, c, s, y);
  gadget_m<M + 1>(a, k, c, s, y);
  gadget_m<M + 2>(a, k, c, s, y);
  gadget_m<M + 3>(a, k, c, s, y);
}

__device__ __forceinline__ uint64_t thread_offset(const TilePass& p, uint32_t tid) {
  uint64_t off = 0;
  for (int j = 0; j < p.ntrun; ++j) off += (uint64_t)(tid & p.trun[j].mask) * p.trun[j].mul;
  return off;
}

// Tile `tile` of the pass; coef: its coefficients in shared memory (COPY: copied there
// from p, otherwise they are in place).
template <bool COPY>
__device__ __forceinline__ void run_tile(float2* __restrict__ psi, const TilePass& p, uint32_t tile, unsigned char* sm,
                                         float* coef) {
  const uint32_t tid = threadIdx.x;
  uint64_t tb = 0;
  for (int j = 0; j < p.nbrun; ++j) tb += (uint64_t)(tile & p.brun[j].mask) * p.brun[j].mul;
  {
    float2* const mine = psi + (tb + thread_offset(p, tid));   // tile index r << kThreadBits | tid is at mine[p.off[r]]
    const uint32_t home = slot(tid) * 8;
    float2 v[kSweepAmps];
#pragma unroll
    for (int r = 0; r < kSweepAmps; ++r) v[r] = mine[p.off[r]];
    if (COPY)
      for (uint32_t e = tid; e < p.ncoef; e += kTileThreads) coef[e] = p.coef[e];
#pragma unroll
    for (int r = 0; r < kSweepAmps; ++r)
      *reinterpret_cast<float2*>(sm + (home ^ slot((uint32_t)r << kThreadBits) * 8)) = v[r];
  }
  __syncthreads();
  for (uint32_t s = 0; s < p.nsweeps; ++s) {
    const TileSweep& w = p.sweep[s];
    uint32_t base = 0;
#pragma unroll
    for (int b = 0; b < kThreadBits; ++b) base += (tid >> b & 1u) * w.mul[b];
    const uint32_t addr = slot(base) * 8;
    float2 a[kSweepAmps];
#pragma unroll
    for (int r = 0; r < kSweepAmps; ++r) a[r] = *reinterpret_cast<const float2*>(sm + (addr ^ w.csw[r]));
    const uint32_t end = w.first + w.count;
    for (uint32_t o = w.first; o < end; ++o) {
      const TileOp& op = p.op[o];
      if (op.kind <= OP_GATE2) {
        if ((tb & op.cg) != op.cg) continue;
        const uint32_t fixed = op.cl & ~op.creg;
        if ((base & fixed) != fixed) continue;
        const uint32_t u = (uint32_t)__cvta_generic_to_shared(coef) + 4 * op.coef;
        if (!op.creg) {
          dense<false>(a, op, u, 0);
        } else {
          uint32_t ok = 0;
#pragma unroll
          for (int r = 0; r < kSweepAmps; ++r) ok |= (((base ^ w.comb[r]) & op.cl) == op.cl ? 1u : 0u) << r;
          dense<true>(a, op, u, ok);
        }
      }
      if (op.kind == OP_GADGET) {
        const uint32_t flip = (uint32_t)(__popcll(tb & op.yzg) + __popc(base & op.yzl)) << 31;
        const uint32_t sb = __float_as_uint(op.s) ^ flip;
        gadget_4m<0>(a, op.k, op.c, sb, op.sgn);
        gadget_4m<4>(a, op.k, op.c, sb, op.sgn);
        gadget_4m<8>(a, op.k, op.c, sb, op.sgn);
        gadget_4m<12>(a, op.k, op.c, sb, op.sgn);
      }
      if (op.kind == OP_DIAG) {
        uint32_t j = 0;
        for (uint32_t q = 0; q < op.nd; ++q) {
          const uint32_t d = op.dpos[q];
          j |= ((d & 0x80u) ? (uint32_t)(tb >> (d & 0x7fu)) & 1u : base >> d & 1u) << q;
        }
        const float2* dg = reinterpret_cast<const float2*>(coef + op.coef);
#pragma unroll
        for (int r = 0; r < kSweepAmps; ++r) {
          const float2 d = dg[j ^ op.jr[r]], x = a[r];
          a[r] = make_float2(d.x * x.x - d.y * x.y, d.x * x.y + d.y * x.x);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < kSweepAmps; ++r) *reinterpret_cast<float2*>(sm + (addr ^ w.csw[r])) = a[r];
    __syncthreads();
  }
  // (computed again instead of kept over the sweeps: registers)
  uint32_t t2;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t2));
  float2* const mine = psi + (tb + thread_offset(p, t2));
  const uint32_t home = slot(t2) * 8;
#pragma unroll
  for (int r = 0; r < kSweepAmps; ++r)
    mine[p.off[r]] = *reinterpret_cast<const float2*>(sm + (home ^ slot((uint32_t)r << kThreadBits) * 8));
}

__global__ void __launch_bounds__(kTileThreads, 4) k_tile_pass(float2* __restrict__ psi, const __grid_constant__ TilePass p) {
  extern __shared__ __align__(16) unsigned char sm[];
  run_tile<true>(psi, p, blockIdx.x, sm, reinterpret_cast<float*>(sm + (sizeof(float2) << kPassBits)));
}

// The same over the tiles of many states: packed passes, copied to shared memory.
__global__ void __launch_bounds__(kTileThreads, 4)
    k_tile_items(float2* __restrict__ pool, const unsigned char* __restrict__ passes, const TileItem* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char sm[];
  const TileItem it = items[blockIdx.x];
  const unsigned char* from = passes + (size_t)it.pass * 16;
  const TilePass& head = *reinterpret_cast<const TilePass*>(from);
  TilePass& p = *reinterpret_cast<TilePass*>(sm + (sizeof(float2) << kPassBits));
  auto copy = [&](void* to, uint32_t bytes) {
    for (uint32_t e = threadIdx.x; e < padded(bytes) / 16; e += kTileThreads)
      static_cast<uint4*>(to)[e] = reinterpret_cast<const uint4*>(from)[e];
    from += padded(bytes);
  };
  const uint32_t ns = head.nsweeps, no = head.nops, nc = head.ncoef;
  copy(&p, kHeadBytes);
  copy(p.sweep, ns * (uint32_t)sizeof(TileSweep));
  copy(p.op, no * (uint32_t)sizeof(TileOp));
  copy(p.coef, nc * (uint32_t)sizeof(float));
  __syncthreads();
  run_tile<false>(pool + it.offset, p, it.tile, sm, p.coef);
}

}  // namespace

cudaError_t launch_tile_items(void* pool, const unsigned char* passes, const qstile::TileItem* items, int nitems,
                              cudaStream_t st) {
  constexpr size_t smem = (sizeof(float2) << kPassBits) + sizeof(TilePass);
  static_assert(4 * (smem + 1024) <= 227 * 1024 && kHeadBytes % 16 == 0, "shared memory");
  static bool attr_done = false;
  if (!attr_done) {
    const cudaError_t e = cudaFuncSetAttribute(k_tile_items, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  k_tile_items<<<nitems, kTileThreads, smem, st>>>(static_cast<float2*>(pool), passes, items);
  return cudaGetLastError();
}

cudaError_t launch_tile_pass(void* amps, const qstile::TilePass& p, cudaStream_t st) {
  static bool attr_done = false;
  if (!attr_done) {
    const cudaError_t e = cudaFuncSetAttribute(k_tile_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmem);
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  k_tile_pass<<<(unsigned)p.ntiles, kTileThreads, kTileSmem, st>>>(static_cast<float2*>(amps), p);
  return cudaGetLastError();
}

}  // namespace qsk
