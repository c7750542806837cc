// Host program for the tile passes of circuits (csrc/qs_tile.h): random circuits of
// every gate kind are scheduled, the passes are run here with the index arithmetic
// of the kernel (csrc/qs_tile.cu), and the state is compared with the gates applied
// one by one.  Also checked: every amplitude belongs to exactly one thread and
// register of a sweep, offsets agree with the tile's bit positions, limits hold.
// Prints the largest difference relative to the largest amplitude, or a fault.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "qs_tile.h"

using namespace qstile;
using cd = std::complex<double>;

struct Circuit {
  std::vector<std::vector<int>> ctrls, targs, paulis;
  std::vector<std::vector<double>> data;
  std::vector<Gate> gates;
};

static int fault(const char* what) {
  std::printf("fault: %s\n", what);
  return 1;
}

static void make(Circuit& c, int n, int count, std::mt19937_64& rng) {
  std::normal_distribution<double> nd;
  c.ctrls.resize(count), c.targs.resize(count), c.paulis.resize(count), c.data.resize(count);
  for (int i = 0; i < count; ++i) {
    std::vector<int> q(n);
    for (int k = 0; k < n; ++k) q[k] = k;
    std::shuffle(q.begin(), q.end(), rng);
    Gate g;
    g.kind = (int)(rng() % 4) % 3;
    const int nt = g.kind == 0 ? 1 + (int)(rng() % 2) : g.kind == 1 ? 1 + (int)(rng() % 6) : (int)(rng() % 7);
    const int nc = g.kind == 0 ? (int)(rng() % 8 ? rng() % 4 : rng() % (n - nt + 1)) : 0;
    c.targs[i].assign(q.begin(), q.begin() + nt);
    c.ctrls[i].assign(q.begin() + nt, q.begin() + nt + nc);
    for (int k = 0; k < nt; ++k) c.paulis[i].push_back((int)(rng() % 4));
    const int m = g.kind == 0 ? 2 << (2 * nt) : 2 << nt;
    for (int k = 0; k < m; ++k) c.data[i].push_back((float)(nd(rng) / (g.kind == 0 ? std::sqrt(2.0 * (1 << nt)) : 1.4)));
    const double phi = -0.5 * nd(rng);
    g.c = std::cos(phi), g.s = std::sin(phi);
    g.ctrls = &c.ctrls[i], g.targs = &c.targs[i], g.paulis = &c.paulis[i], g.data = c.data[i].data();
    for (int k = 0; k < nt + nc; ++k) g.qmask |= 1ull << q[k];
    c.gates.push_back(g);
  }
}

static void direct(const Gate& g, std::vector<cd>& a) {
  std::vector<cd> o(a);
  const int nt = (int)g.targs->size();
  for (size_t i = 0; i < a.size(); ++i) {
    int j = 0;
    size_t rest = i;
    for (int k = 0; k < nt; ++k) {
      j |= (int)(i >> (*g.targs)[k] & 1) << k;
      rest &= ~((size_t)1 << (*g.targs)[k]);
    }
    if (g.kind == 0) {
      bool ok = true;
      for (int c : *g.ctrls) ok = ok && (i >> c & 1);
      if (!ok) continue;
      cd s = 0;
      for (int l = 0; l < (1 << nt); ++l) {
        size_t x = rest;
        for (int k = 0; k < nt; ++k)
          if (l >> k & 1) x |= (size_t)1 << (*g.targs)[k];
        s += cd(g.data[2 * ((j << nt) + l)], g.data[2 * ((j << nt) + l) + 1]) * a[x];
      }
      o[i] = s;
    } else if (g.kind == 1) {
      o[i] = a[i] * cd(g.data[2 * j], g.data[2 * j + 1]);
    } else {
      uint64_t xy = 0, yz = 0;
      int ny = 0;
      for (int k = 0; k < nt; ++k) {
        const int p = (*g.paulis)[k];
        if (p == 1 || p == 2) xy |= 1ull << (*g.targs)[k];
        if (p >= 2) yz |= 1ull << (*g.targs)[k];
        ny += p == 2;
      }
      static const cd ipow[4] = {{1, 0}, {0, 1}, {-1, 0}, {0, -1}};
      const size_t k = i ^ xy;
      o[i] = g.c * a[i] + ipow[(ny + 1) & 3] * g.s * (parity(k & yz) ? -1.0 : 1.0) * a[k];
    }
  }
  a.swap(o);
}

static cd entry(const float* d, int e) {
  d += 4 * e;
  return d[0] == d[1] && d[2] == -d[3] ? cd(d[0], d[3]) : cd(NAN, NAN);
}

static int run(const TilePass& p, std::vector<cd>& psi) {
  constexpr uint32_t kAmps = 1u << kPassBits, kThreads = 1u << kThreadBits;
  if (p.ncoef > kMaxCoef || p.nops > kMaxOps || p.nsweeps > kMaxOps) return fault("limits");
  for (uint64_t tile = 0; tile < p.ntiles; ++tile) {
    uint64_t tb = 0;
    for (int j = 0; j < p.nbrun; ++j) tb += (uint64_t)((uint32_t)tile & p.brun[j].mask) * p.brun[j].mul;
    std::vector<cd> sm(kAmps);
    std::vector<uint64_t> where(kAmps);
    for (uint32_t i = 0; i < kAmps; ++i) {
      uint64_t o = tb, g = tb;
      const uint32_t tid = i % kThreads, r = i / kThreads;
      for (int j = 0; j < p.ntrun; ++j) o += (uint64_t)(tid & p.trun[j].mask) * p.trun[j].mul;
      o += p.off[r];
      for (int b = 0; b < kPassBits; ++b) {
        if (tb >> p.P[b] & 1) return fault("tile offset");
        if (i >> b & 1) g |= 1ull << p.P[b];
      }
      if (o != g || o >= psi.size()) return fault("offset");
      if ((slot(tid) ^ slot(r << kThreadBits)) != slot(i)) return fault("slot");
      where[i] = g;
      sm[slot(i)] = psi[g];
    }
    for (uint32_t s = 0; s < p.nsweeps; ++s) {
      const TileSweep& w = p.sweep[s];
      std::vector<char> seen(kAmps);
      for (uint32_t t = 0; t < kThreads; ++t) {
        uint32_t base = 0;
        for (int b = 0; b < kThreadBits; ++b) base += (t >> b & 1) * w.mul[b];
        cd v[kSweepAmps], old[kSweepAmps];
        for (int r = 0; r < kSweepAmps; ++r) {
          const uint32_t at = slot(base) * 8 ^ w.csw[r];
          if (at % 8 || at / 8 >= kAmps || seen[at / 8]) return fault("cosets");
          seen[at / 8] = 1;
          v[r] = sm[at / 8];
        }
        for (uint32_t o = w.first; o < w.first + w.count; ++o) {
          const TileOp& op = p.op[o];
          const float* d = p.coef + op.coef;
          if (op.coef % 4) return fault("alignment");
          std::copy(v, v + kSweepAmps, old);
          for (int r = 0; r < kSweepAmps; ++r) {
            if (op.kind <= OP_GATE2 && ((tb & op.cg) != op.cg || ((base ^ w.comb[r]) & op.cl) != op.cl)) continue;
            if (op.kind == OP_GATE1) {
              const int j = r >> op.k & 1, r0 = r & ~(1 << op.k);
              v[r] = entry(d, 2 * j) * old[r0] + entry(d, 2 * j + 1) * old[r0 | 1 << op.k];
            } else if (op.kind == OP_GATE2) {
              static const int K0[6] = {0, 0, 0, 1, 1, 2}, K1[6] = {1, 2, 3, 2, 3, 3};
              const int k0 = K0[op.k], k1 = K1[op.k], j = (r >> k0 & 1) | (r >> k1 & 1) << 1;
              const int r0 = r & ~(1 << k0) & ~(1 << k1);
              v[r] = 0;
              for (int l = 0; l < 4; ++l)
                v[r] += entry(d, 4 * j + l) * old[r0 | (l & 1) << k0 | (l >> 1) << k1];
            } else if (op.kind == OP_GADGET) {
              const int sg = parity(tb & op.yzg) ^ parity(base & op.yzl) ^ parity(op.sgn & (uint32_t)r);
              const double f = sg ? -op.s : op.s;
              v[r] = (double)op.c * old[r] + (op.k >> 4 ? cd(0, f) : cd(f, 0)) * old[r ^ (op.k & 15)];
            } else {
              uint32_t j = 0;
              for (uint32_t q = 0; q < op.nd; ++q)
                j |= (op.dpos[q] & 0x80 ? (uint32_t)(tb >> (op.dpos[q] & 0x7f)) & 1u : base >> op.dpos[q] & 1u) << q;
              j ^= op.jr[r];
              v[r] = old[r] * cd(d[2 * j], d[2 * j + 1]);
            }
          }
        }
        for (int r = 0; r < kSweepAmps; ++r) sm[(slot(base) * 8 ^ w.csw[r]) / 8] = v[r];
      }
    }
    for (uint32_t i = 0; i < kAmps; ++i) psi[where[i]] = sm[slot(i)];
  }
  return 0;
}

int main() {
  std::mt19937_64 rng(5);
  double worst = 0;
  for (int trial = 0; trial < 24; ++trial) {
    const int n = kPassBits + trial % 4;
    Circuit c;
    make(c, n, 60, rng);
    std::normal_distribution<double> nd;
    std::vector<cd> a((size_t)1 << n), b;
    for (auto& x : a) x = {nd(rng), nd(rng)};
    b = a;
    std::vector<TilePass> passes;
    for (const Gate& g : c.gates) {
      if (!fits(g, n)) return fault("fits");
      direct(g, a);
    }
    std::vector<unsigned char> packed;
    std::vector<size_t> at;
    build_passes(c.gates, n, [&](const TilePass& p) {
      at.push_back(packed.size());
      pack(p, &packed);
    });
    for (size_t a : at) {
      passes.emplace_back();
      unpack(packed.data() + a, &passes.back());
    }
    size_t ops = 0;
    for (const TilePass& p : passes) {
      ops += p.nops;
      if (run(p, b)) return 1;
    }
    if (ops != c.gates.size()) return fault("gates lost");
    double e = 0, m = 0;
    for (size_t i = 0; i < a.size(); ++i) {
      e = std::max(e, std::abs(a[i] - b[i]));
      m = std::max(m, std::abs(a[i]));
    }
    worst = std::max(worst, e / m);
  }
  std::printf("%.3g\n", worst);
  return 0;
}
