// Tile passes of circuits: host side (no CUDA dependency; tests/host/tile_check.cpp
// compiles it with g++ alone).
//
// A pass holds a tile of 2^kPassBits amplitudes in shared memory, reads and writes
// the state once and applies many gates in between.  The tile's index bits are the
// kPassLow lowest qubits (runs of 128 bytes) and up to kPassHigh more, chosen for
// the gates: a gate fits if the qubits it flips (targets of dense gates, X and Y
// factors of gadgets) are among them; controls, Z factors and diagonals only read
// index bits and fit anywhere.
//
// Inside a pass gates are grouped into sweeps.  A sweep's gates flip indices along
// at most kSweepDim directions of GF(2)^kPassBits (a target's unit vector, a
// gadget's flip mask); a thread holds the 2^kSweepDim amplitudes of one coset of
// their span in registers, reads them once and applies all of the sweep's gates.
// Gates that share no qubit commute exactly, so both levels take gates past
// skipped ones when nothing in between touches their qubits.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cstring>
#include <utility>
#include <vector>

#ifdef __CUDACC__
#define QT_HD __host__ __device__
#else
#define QT_HD
#endif

namespace qstile {

constexpr int kPassBits = 12;      // 32 KB of complex64
constexpr int kPassLow = 4;
constexpr int kPassHigh = kPassBits - kPassLow;
constexpr int kSweepDim = 4;
constexpr int kSweepAmps = 1 << kSweepDim;
constexpr int kThreadBits = kPassBits - kSweepDim;
constexpr int kMaxOps = 24;
constexpr int kMaxCoef = 1024;
// Gates in a row that a pass looks past without taking one: keeps schedules linear in
// the gates where some qubit never gets blocked (100,000 gates on 20 of 29 qubits: 11.7 s
// without it, 0.1 s with it; the passes are the same).
constexpr int kLookAhead = 256;

enum { OP_GATE1 = 0, OP_GATE2 = 1, OP_GADGET = 2, OP_DIAG = 3 };

struct TileOp {
  uint64_t cg, yzg;                // control / sign masks on qubits outside the tile
  uint32_t cl, yzl;                // and on tile bits
  uint32_t sgn;                    // gadget: bit k = parity(yzl & direction k)
  uint32_t coef;                   // offset of the coefficients, a multiple of four
  uint32_t kind;
  uint32_t k;                      // gate1: register bit; gate2: pair index; gadget: m | imaginary << 4
  uint32_t creg;                   // controls that differ inside a coset
  uint32_t nd;                     // diagonal: targets
  uint8_t dpos[8];                 // their tile bits, or 0x80 | qubit
  uint8_t jr[kSweepAmps];          // diagonal: entry index bits of comb[r]
  float c, s;                      // gadget
};

struct TileSweep {
  uint32_t csw[kSweepAmps];        // shared-memory byte offset (xor) of register r
  uint32_t mul[kThreadBits];       // 2^(tile bit of thread-index bit b)
  uint16_t comb[kSweepAmps];       // tile index xor of register r
  uint32_t first, count;           // ops
};

// Scatter of index bits: run j moves the bits in mask by a factor of two's power.
struct TileRun {
  uint32_t mask, mul;
};

struct TilePass {
  uint64_t ntiles;
  uint64_t off[kSweepAmps];        // qubit offset of tile index r << kThreadBits
  TileRun brun[kPassBits + 1];     // tile number -> bits outside the tile
  TileRun trun[kThreadBits];       // thread-index bits 0..kThreadBits-1 -> tile bits of the same number
  int8_t P[kPassBits];             // qubit of tile bit b, ascending; 0..kPassLow-1 first
  uint8_t nbrun, ntrun;
  uint32_t nsweeps, nops, ncoef;
  alignas(16) TileSweep sweep[kMaxOps];
  alignas(16) TileOp op[kMaxOps];
  alignas(16) float coef[kMaxCoef];
};

// One block of a launch over many states: a tile of a pass.
struct TileItem {
  uint64_t offset;                 // of the state's first amplitude
  uint32_t pass, tile;             // pass: where its packed form starts, in units of 16 bytes
};

QT_HD constexpr uint32_t padded(uint32_t bytes) { return (bytes + 15) & ~15u; }
constexpr uint32_t kHeadBytes = offsetof(TilePass, sweep);

// Appends a pass without its unused parts: head, sweeps, operations, coefficients,
// each padded to 16 bytes (about 2 KB where the whole struct has 8.7).
inline void pack(const TilePass& p, std::vector<unsigned char>* out) {
  auto put = [&](const void* from, uint32_t bytes) {
    const unsigned char* f = static_cast<const unsigned char*>(from);
    out->insert(out->end(), f, f + bytes);
    out->resize(padded((uint32_t)bytes) - bytes + out->size());
  };
  put(&p, kHeadBytes);
  put(p.sweep, (uint32_t)sizeof(TileSweep) * p.nsweeps);
  put(p.op, (uint32_t)sizeof(TileOp) * p.nops);
  put(p.coef, (uint32_t)sizeof(float) * p.ncoef);
}

// The pass packed at `from`.
inline void unpack(const unsigned char* from, TilePass* p) {
  auto get = [&](void* to, uint32_t bytes) {
    std::memcpy(to, from, bytes);
    from += padded(bytes);
  };
  get(p, kHeadBytes);
  get(p->sweep, (uint32_t)sizeof(TileSweep) * p->nsweeps);
  get(p->op, (uint32_t)sizeof(TileOp) * p->nops);
  get(p->coef, (uint32_t)sizeof(float) * p->ncoef);
}

// Shared-memory slot of tile index i: the bank bits 0..3 (8-byte words) fold in
// every higher bit, so that lanes along any four suitable bits meet each bank once.
QT_HD constexpr uint32_t slot(uint32_t i) { return i ^ (((i >> 4) ^ (i >> 8) ^ (i >> 12)) & 15u); }

struct Gate {
  int kind = 0;                    // 0 dense, 1 diagonal, 2 gadget
  const std::vector<int>*ctrls = nullptr, *targs = nullptr, *paulis = nullptr;
  const double* data = nullptr;
  double c = 1.0, s = 0.0;         // gadget: cos and sin of phi = -theta / 2
  uint64_t qmask = 0;
};

// Qubits that the gate flips.
inline uint64_t flips(const Gate& g) {
  uint64_t m = 0;
  if (g.kind == 0)
    for (int t : *g.targs) m |= 1ull << t;
  if (g.kind == 2)
    for (size_t q = 0; q < g.targs->size(); ++q)
      if ((*g.paulis)[q] == 1 || (*g.paulis)[q] == 2) m |= 1ull << (*g.targs)[q];
  return m;
}

// Floats of a gate's coefficients: a matrix entry is (re, re, -im, im).
inline int coefs(const Gate& g) {
  return g.kind == 0 ? 4 << (2 * g.targs->size()) : g.kind == 1 ? 2 << g.targs->size() : 0;
}

// Whether tile passes of a state of nq qubits can hold the gate.
inline bool fits(const Gate& g, int nq) {
  if (nq < kPassBits) return false;
  if (g.kind == 0 && g.targs->size() > 2) return false;
  return __builtin_popcountll(flips(g) >> kPassLow) <= kPassHigh;
}

inline int parity(uint64_t x) { return __builtin_popcountll(x) & 1; }

// Bank bits of a tile index.
inline uint32_t bank(uint32_t i) { return slot(i) & 15u; }

inline void put_entry(float* d, const double* m) {
  d[0] = d[1] = (float)m[0];
  d[2] = (float)-m[1];
  d[3] = (float)m[1];
}

// The sweep of the pass's ops [first, first + count) and their directions
// (unit vectors of dense targets in `unit`, gadget masks in `masks`; `ctl`: tile bits
// that control a gate of the sweep).
inline void finish_sweep(TilePass& p, TileSweep& sw, const std::vector<Gate>& gs, const std::vector<uint32_t>& loc,
                         uint32_t unit, const std::vector<uint32_t>& masks, uint32_t ctl) {
  // basis in reduced echelon form: dense targets first, as unit vectors
  uint32_t v[kSweepDim], piv[kSweepDim];
  int dim = 0;
  uint32_t pivots = 0;
  for (int b = 0; b < kPassBits; ++b)
    if (unit >> b & 1) {
      v[dim] = 1u << b;
      piv[dim++] = b;
      pivots |= 1u << b;
    }
  for (uint32_t x : masks) {
    for (int k = 0; k < dim; ++k)
      if (x >> piv[k] & 1) x ^= v[k];
    if (!x) continue;
    const uint32_t b = 31 - __builtin_clz(x);
    for (int k = 0; k < dim; ++k)
      if (v[k] >> b & 1) v[k] ^= x;          // never a dense target's: x is zero there, and so is their bit b
    v[dim] = x;
    piv[dim++] = b;
    pivots |= 1u << b;
  }
  // fill with the highest bits that are free, those of no control first
  for (int b = 2 * kPassBits - 1; dim < kSweepDim; --b) {
    const int avoid = b >= kPassBits;
    if (avoid) b -= kPassBits;
    if ((pivots >> b & 1) || (avoid && (ctl >> b & 1))) {
      if (avoid) b += kPassBits;
      continue;
    }
    for (int k = 0; k < dim; ++k)
      if (v[k] >> b & 1) v[k] ^= 1u << b;
    v[dim] = 1u << b;
    piv[dim++] = b;
    pivots |= 1u << b;
    if (avoid) b += kPassBits;
  }
  for (int r = 0; r < kSweepAmps; ++r) {
    uint32_t c = 0;
    for (int k = 0; k < kSweepDim; ++k)
      if (r >> k & 1) c ^= v[k];
    sw.comb[r] = (uint16_t)c;
    sw.csw[r] = slot(c) * 8;
  }
  // thread-index bits: first four tile bits with independent banks (the lanes of a
  // half warp), then the others in order
  uint32_t used = pivots, span[16] = {0};
  int nb = 0, have = 1;
  for (int b = 0; b < kPassBits && nb < 4; ++b) {
    if (used >> b & 1) continue;
    const uint32_t k = bank(1u << b);
    bool in = false;
    for (int i = 0; i < have; ++i) in = in || span[i] == k;
    if (in) continue;
    for (int i = 0; i < have; ++i) span[have + i] = span[i] ^ k;
    have *= 2;
    sw.mul[nb++] = 1u << b;
    used |= 1u << b;
  }
  for (int b = 0; b < kPassBits; ++b)
    if (!(used >> b & 1)) sw.mul[nb++] = 1u << b;
  auto reg = [&](uint32_t x) {               // register index of a flip mask in the span
    uint32_t m = 0;
    for (int k = 0; k < kSweepDim; ++k)
      if (x >> piv[k] & 1) m |= 1u << k;
    return m;
  };
  auto tile_mask = [&](uint64_t q) {
    uint32_t m = 0;
    for (int b = 0; b < kPassBits; ++b)
      if (q >> p.P[b] & 1) m |= 1u << b;
    return m;
  };
  uint64_t inside = 0;
  for (int b = 0; b < kPassBits; ++b) inside |= 1ull << p.P[b];
  for (int o = sw.first; o < sw.first + sw.count; ++o) {
    const Gate& g = gs[o];
    TileOp& op = p.op[o];
    std::memset(&op, 0, sizeof(op));
    op.coef = p.ncoef;
    if (g.kind == 0) {
      uint64_t cm = 0;
      for (int c : *g.ctrls) cm |= 1ull << c;
      op.cg = cm & ~inside;
      op.cl = tile_mask(cm);
      for (int r = 1; r < kSweepAmps; ++r) op.creg |= sw.comb[r] & op.cl;
      const int n = (int)g.targs->size();
      float* d = p.coef + p.ncoef;
      if (n == 1) {
        op.kind = OP_GATE1;
        op.k = (uint32_t)__builtin_ctz(reg(1u << loc[(*g.targs)[0]]));
        for (int e = 0; e < 4; ++e) put_entry(d + 4 * e, g.data + 2 * e);
      } else {
        op.kind = OP_GATE2;
        int k0 = __builtin_ctz(reg(1u << loc[(*g.targs)[0]])), k1 = __builtin_ctz(reg(1u << loc[(*g.targs)[1]]));
        const bool sw2 = k0 > k1;            // matrix bit 0 on the lower register bit
        if (sw2) std::swap(k0, k1);
        op.k = (uint32_t)(k0 == 0 ? k1 - 1 : k0 == 1 ? k1 + 1 : 5);   // 01 02 03 12 13 23
        auto perm = [&](int j) { return sw2 ? (j & 1) << 1 | j >> 1 : j; };
        for (int j = 0; j < 4; ++j)
          for (int l = 0; l < 4; ++l) put_entry(d + 4 * (4 * j + l), g.data + 2 * (4 * perm(j) + perm(l)));
      }
      p.ncoef += (uint32_t)coefs(g);
    } else if (g.kind == 1) {
      op.kind = OP_DIAG;
      op.nd = (uint32_t)g.targs->size();
      for (uint32_t q = 0; q < op.nd; ++q) {
        const int t = (*g.targs)[q];
        op.dpos[q] = (uint8_t)(inside >> t & 1 ? loc[t] : 0x80 | t);
        if (inside >> t & 1)
          for (int r = 0; r < kSweepAmps; ++r) op.jr[r] |= (uint8_t)((sw.comb[r] >> loc[t] & 1) << q);
      }
      for (int e = 0; e < coefs(g); ++e) p.coef[p.ncoef + e] = (float)g.data[e];
      p.ncoef += (uint32_t)coefs(g);
    } else {
      op.kind = OP_GADGET;
      uint64_t xy = 0, yz = 0;
      int ny = 0;
      for (size_t q = 0; q < g.targs->size(); ++q) {
        const int c = (*g.paulis)[q];
        if (c == 1 || c == 2) xy |= 1ull << (*g.targs)[q];
        if (c == 2 || c == 3) yz |= 1ull << (*g.targs)[q];
        ny += c == 2;
      }
      const uint32_t m = reg(tile_mask(xy));
      op.yzg = yz & ~inside;
      op.yzl = tile_mask(yz);
      for (int k = 0; k < kSweepDim; ++k) op.sgn |= (uint32_t)parity(v[k] & op.yzl) << k;
      // exp(i phi P): c a_i + s i^q a_j, j = i ^ xy, with the sign of parity(j & yz):
      // register 0 pairs with register m
      const int q = (ny + 1 + 2 * parity(sw.comb[m] & op.yzl)) & 3;
      op.k = m | (uint32_t)(q & 1) << 4;
      op.c = (float)g.c;
      op.s = (float)(q >= 2 ? -g.s : g.s);
    }
  }
}

// Passes that apply the gates (each fits()) in an equivalent order, handed to emit one
// by one.
template <typename Emit>
inline void build_passes(const std::vector<Gate>& gates, int nq, const Emit& emit) {
  std::vector<int> left, rest;              // left: from `begin` on
  size_t begin = 0;
  for (int i = 0; i < (int)gates.size(); ++i) left.push_back(i);
  std::vector<uint64_t> ahead(gates.size());   // qubits of this gate and all after it
  for (size_t i = gates.size(); i-- > 0;) ahead[i] = gates[i].qmask | (i + 1 < gates.size() ? ahead[i + 1] : 0);
  while (begin < left.size()) {
    std::vector<int> take;
    uint64_t tile = (1ull << kPassLow) - 1, blocked = 0;
    int ncoef = 0;
    rest.clear();
    // until every gate ahead meets a skipped one, or kLookAhead gates in a row have
    size_t at = begin;
    int skipped = 0;
    for (; at < left.size() && (blocked == 0 || (ahead[left[at]] & ~blocked)) && skipped < kLookAhead &&
           (int)take.size() < kMaxOps;
         ++at) {
      const Gate& g = gates[left[at]];
      const uint64_t t = tile | flips(g);
      if (!(g.qmask & blocked) && __builtin_popcountll(t) <= kPassBits && ncoef + coefs(g) <= kMaxCoef) {
        take.push_back(left[at]);
        tile = t;
        ncoef += coefs(g);
        skipped = 0;
      } else {
        blocked |= g.qmask;
        rest.push_back(left[at]);
        ++skipped;
      }
    }
    begin = at - rest.size();               // the skipped gates, then those not looked at
    for (size_t i = 0; i < rest.size(); ++i) left[begin + i] = rest[i];
    for (int q = 0; __builtin_popcountll(tile) < kPassBits; ++q) tile |= 1ull << q;
    TilePass p;
    std::memset(static_cast<void*>(&p), 0, sizeof(p));
    p.ntiles = 1ull << (nq - kPassBits);
    std::vector<uint32_t> loc(64, 0);
    for (int q = 0, b = 0; q < nq; ++q)
      if (tile >> q & 1) {
        p.P[b] = (int8_t)q;
        loc[q] = (uint32_t)b++;
      }
    for (int r = 0; r < kSweepAmps; ++r)
      for (int b = 0; b < kSweepDim; ++b)
        if (r >> b & 1) p.off[r] |= 1ull << p.P[kThreadBits + b];
    // tile bits b with equal P[b] - b, and the qubits between tile bits, move together
    for (int b = 0; b < kThreadBits; ++b) {
      if (b == 0 || p.P[b] != p.P[b - 1] + 1) p.trun[p.ntrun++] = TileRun{0, 1u << (p.P[b] - b)};
      p.trun[p.ntrun - 1].mask |= 1u << b;
    }
    for (int q = 0, j = 0, below = 0, last = -2; q < nq; ++q) {
      if (tile >> q & 1) {
        ++below;
        continue;
      }
      if (below != last) p.brun[p.nbrun++] = TileRun{0, 1u << below};
      last = below;
      p.brun[p.nbrun - 1].mask |= 1u << j++;
    }
    // sweeps
    std::vector<Gate> gs;                     // in the order of p.op
    while (!take.empty()) {
      TileSweep& sw = p.sweep[p.nsweeps++];
      sw.first = (uint32_t)gs.size();
      std::vector<int> later;
      std::vector<uint32_t> masks, ech;       // gadget masks; echelon form of all directions
      uint32_t unit = 0, flipped = 0, ctl = 0;
      blocked = 0;
      for (int i : take) {
        const Gate& g = gates[i];
        bool ok = !(g.qmask & blocked);
        if (ok) {
          uint32_t m = 0, cl = 0;
          const uint64_t f = flips(g);
          for (int b = 0; b < kPassBits; ++b)
            if (f >> p.P[b] & 1) m |= 1u << b;
          if (g.kind == 0)
            for (int c : *g.ctrls)
              if (tile >> c & 1) cl |= 1u << loc[c];
          std::vector<uint32_t> dirs, e2 = ech;
          if (g.kind == 0)
            for (int t : *g.targs) dirs.push_back(1u << loc[t]);
          else if (m)
            dirs.push_back(m);
          for (uint32_t x : dirs) {
            for (uint32_t v : e2)
              if ((x ^ v) < x) x ^= v;
            if (x) e2.push_back(x);
          }
          // controls that no direction of the sweep flips are equal over a thread's
          // amplitudes
          ok = (int)e2.size() <= kSweepDim && !((flipped | m) & (ctl | cl));
          if (ok) {
            ech = e2;
            flipped |= m;
            ctl |= cl;
            if (g.kind == 0)
              unit |= m;
            else if (m)
              masks.push_back(m);
          }
        }
        if (ok) {
          gs.push_back(g);
          ++sw.count;
        } else {
          blocked |= g.qmask;
          later.push_back(i);
        }
      }
      take.swap(later);
      p.nops = (uint32_t)gs.size();
      finish_sweep(p, sw, gs, loc, unit, masks, ctl);
    }
    emit(p);
  }
}

}  // namespace qstile
