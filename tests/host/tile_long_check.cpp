// Time to schedule long circuits (csrc/qs_tile.h): 100,000 gates on all qubits, on some
// of them, and with a qubit that only the last gate touches.  Prints the three times and
// the passes, or a fault when gates are lost.
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <random>

#include "qs_tile.h"

using namespace qstile;

int main() {
  constexpr int n = 29, G = 100000;
  for (int kind = 0; kind < 3; ++kind) {
    std::mt19937 rng(3);
    const int used = kind == 0 ? n : kind == 1 ? 20 : n - 1;
    std::vector<std::vector<int>> ctrls(G), targs(G), paulis(G);
    std::vector<double> data(64, 0.5);
    std::vector<Gate> gates;
    std::vector<int> q(used);
    for (int k = 0; k < used; ++k) q[k] = k;
    for (int i = 0; i < G; ++i) {
      std::shuffle(q.begin(), q.end(), rng);
      const int k = rng() % 3;
      Gate g;
      const bool phase = kind == 0 && i >= G - 60;       // global phases at the end
      g.kind = phase || k == 2 ? 2 : 0;
      const int nt = phase ? 0 : k == 0 ? 1 : k == 1 ? 1 + rng() % 2 : 1 + rng() % 6, nc = k == 1 && !phase ? rng() % 4 : 0;
      targs[i].assign(q.begin(), q.begin() + nt);
      if (kind == 2 && i == G - 1) targs[i].assign(nt, n - 1), targs[i].resize(1);
      ctrls[i].assign(q.begin() + nt, q.begin() + nt + nc);
      for (size_t j = 0; j < targs[i].size(); ++j) paulis[i].push_back(1 + rng() % 3);
      g.ctrls = &ctrls[i], g.targs = &targs[i], g.paulis = &paulis[i], g.data = data.data();
      for (int t : targs[i]) g.qmask |= 1ull << t;
      for (int c : ctrls[i]) g.qmask |= 1ull << c;
      gates.push_back(g);
    }
    size_t ops = 0, passes = 0;
    const auto t0 = std::chrono::steady_clock::now();
    build_passes(gates, n, [&](const TilePass& p) {
      ops += p.nops;
      ++passes;
    });
    const double s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (ops != gates.size()) return std::printf("gates lost\n"), 1;
    std::printf("%.4f %zu\n", s, passes);
  }
  return 0;
}
