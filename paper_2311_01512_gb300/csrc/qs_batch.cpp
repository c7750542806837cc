// Batched engine (C ABI, include/qs.h): many independent statevectors with
// their own circuits, run by one persistent kernel launch (qs_batch_kernels.cu)
// that is captured once in a CUDA graph and replayed.
//
// Scheduling: states are ordered by estimated work (amplitudes x operation costs),
// largest first, and CTAs take them from a shared counter, so the long states
// start early and the short ones fill the gaps (longest-processing-time
// order).  A state with more than a CTA's share of the work would outlast the
// rest; such heavy states are shared by the CTAs of a cluster.  The launch shape (threads per CTA, CTAs per SM, and with it the
// largest state kept in shared memory) is chosen by timing every candidate on
// the batch itself.
//
// States larger than shared memory are cut into segments (cache blocking):
// consecutive operations are grouped while the qubits they pair (dense
// targets, gadget X/Y qubits) together with the five lowest qubits fit in a
// tile of L qubits; the kernel then moves each tile through shared memory once
// per segment instead of moving the state once per operation.
//
// complex64 states of at least a tile of qs_tile.h whose operations fit its passes
// can take those instead: launch k runs the k-th pass of every such state, one block
// per tile, while a second branch of the graph runs the other states.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_runtime.h>

#include "qs.h"
#include "qs_handle.h"
#include "qs_alloc.h"
#include "qs_internal.h"
#include "qs_batch_plan.h"
#include "qs_tile.h"

struct qs_batch {
  qs_prec prec = QS_C64;
  cudaStream_t stream = nullptr;
  std::vector<int> nq;          // storage qubits (2N for a density matrix)
  std::vector<int> nlog;        // N: the qubits operations name
  std::vector<int> dens;        // density matrix (Choi vector) or statevector
  std::vector<size_t> offset;  // amplitudes
  size_t pool_amps = 0;
  void* pool = nullptr;
  std::vector<std::vector<qsk::BatchOp>> progs;
  std::vector<std::vector<double>> consts;   // per state; BatchOp::coff indexes it until compile
  qsk::BatchState* d_states = nullptr;
  qsk::BatchSeg* d_segs = nullptr;
  qsk::BatchXlat* d_xlat = nullptr;
  int* d_order = nullptr;
  qsk::BatchOp* d_ops = nullptr;
  double* d_consts = nullptr;
  int* d_counter = nullptr;
  // tile passes: packed descriptors, blocks of launch k at [level[k], level[k + 1])
  unsigned char* d_passes = nullptr;
  qstile::TileItem* d_items = nullptr;
  std::vector<int> level;
  long num_segs = 0;
  int wide = 0;                 // some operation is dense on 3 or 4 targets
  int threads = 256, ctas = 0, smem_qubits = -1;
  int cluster = 1;              // heavy states (first in the order) are shared by clusters of CTAs
  cudaStream_t capture_stream = nullptr;  // own stream for recording (the caller's may be the legacy stream)
  cudaStream_t branch_stream = nullptr;   // and for the graph's second branch
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  bool compiled = false;
  long total_ops = 0;
  float best_ms = 0.f;
};

namespace {

void free_device(qs_batch* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  for (void* p : {(void*)b->d_states, (void*)b->d_segs, (void*)b->d_xlat, (void*)b->d_order, (void*)b->d_ops,
                  (void*)b->d_consts, (void*)b->d_counter, (void*)b->d_passes, (void*)b->d_items})
    if (p) cudaFree(p);
  b->d_consts = nullptr;
  b->exec = nullptr;
  b->graph = nullptr;
  b->d_states = nullptr;
  b->d_segs = nullptr;
  b->d_xlat = nullptr;
  b->d_order = nullptr;
  b->d_ops = nullptr;
  b->d_counter = nullptr;
  b->d_passes = nullptr;
  b->d_items = nullptr;
  b->level.clear();
  b->compiled = false;
}

qs_status check_state(const qs_batch* b, int s) {
  if (!b || s < 0 || s >= (int)b->nq.size()) return QS_ERR_ARG;
  return QS_OK;
}

// one operation on storage qubits, with its nc constants
qs_status add(qs_batch* b, int s, qsk::BatchOp op, const double* c, size_t nc) {
  op.coff = b->consts[s].size();
  b->consts[s].insert(b->consts[s].end(), c, c + nc);
  b->progs[s].push_back(op);
  b->compiled = false;
  return QS_OK;
}

// dense operation on storage targets t (matrix bit q on t[q]) with storage controls c
qs_status add_dense(qs_batch* b, int s, const std::vector<int>& c, const std::vector<int>& t, const double* mat) {
  qsk::BatchOp op{};
  op.kind = 0;
  op.n = (int)t.size();
  std::vector<int> ins(t);
  for (int q = 0; q < op.n; ++q) op.t[q] = t[q];
  for (int q : c) {
    op.ctrl |= 1u << q;
    ins.push_back(q);
  }
  if (ins.size() > 7) return QS_ERR_TOO_MANY_TARGETS;
  std::sort(ins.begin(), ins.end());
  op.nins = (int)ins.size();
  for (int i = 0; i < op.nins; ++i) op.ins[i] = (int8_t)ins[i];
  return add(b, s, op, mat, (size_t)2 << (2 * op.n));
}

// Superoperator of a channel on the Choi vector as a dense operation on
// (t, t + N) (one qubit) or (t1, t2, t1 + N, t2 + N) (two qubits): member m
// has bit q of m on the q-th of those positions; S (real, row-major, d x d)
// gives new beta_m = sum_k S[m][k] beta_k.
qs_status add_superop(qs_batch* b, int s, const std::vector<int>& targs, const std::vector<double>& S) {
  const int n = (int)targs.size(), d = 1 << (2 * n);
  std::vector<int> t(targs);
  for (int q = 0; q < n; ++q) t.push_back(targs[q] + b->nlog[s]);
  std::vector<double> m((size_t)2 * d * d, 0.0);
  for (int i = 0; i < d * d; ++i) m[2 * i] = S[i];
  return add_dense(b, s, {}, t, m.data());
}

qs_status check_density(const qs_batch* b, int s) {
  if (check_state(b, s) != QS_OK) return QS_ERR_ARG;
  return b->dens[s] ? QS_OK : QS_ERR_NOT_DENSMATR;
}

qs_status check_prob(double p) { return (p >= 0.0 && p <= 1.0) ? QS_OK : QS_ERR_ARG; }

// One-qubit channels in the paper's Choi-vector form: members 00 and 11 (bits
// t, t + N) mix as f0 self + f1 other; 01 and 10 as f2 self + f3 other.
qs_status add_channel1(qs_batch* b, int s, int t, double f0, double f1, double f2, double f3) {
  if (check_density(b, s) != QS_OK) return check_density(b, s);
  qs_status st = qsapi::check_qubits(b->nlog[s], &t, 1, nullptr, 0);
  if (st != QS_OK) return st;
  return add_superop(b, s, {t}, qsbatch::channel1_superop(f0, f1, f2, f3));
}

int smem_qubits_for(qs_prec prec, int ctas_per_sm) {
  const size_t per_cta = std::min<size_t>(200 * 1024 / ctas_per_sm, 200 * 1024);
  const size_t amp = prec == QS_C128 ? 16 : 8;
  int q = 0;
  while (((size_t)1 << (q + 1)) * amp <= per_cta) ++q;
  return q;
}

// ---- segment plans (for one tile size L) ------------------------------------
struct Plan {
  int L = -1;
  int cluster = 1;                    // CTAs that share a heavy state
  std::vector<qsk::BatchState> states;
  std::vector<qsk::BatchSeg> segs;
  std::vector<qsk::BatchXlat> xlat;   // parallel to the operations
  qsk::BatchState* d_states = nullptr;
  qsk::BatchSeg* d_segs = nullptr;
  qsk::BatchXlat* d_xlat = nullptr;
  void release() {
    for (void* p : {(void*)d_states, (void*)d_segs, (void*)d_xlat})
      if (p) cudaFree(p);
    d_states = nullptr;
    d_segs = nullptr;
    d_xlat = nullptr;
  }
};

// Least qubits of a heavy state: eight tiles (the largest cluster) of 2^8 amplitudes.
constexpr int kHeavyMinQubits = 11;

// Segments of every state larger than 2^L amplitudes (qs_batch_plan.h); with
// clusters, heavy states in tiles small enough for one per CTA of a cluster.
void build_plan(Plan& P, int L, int cluster, const std::vector<int>& nq, const std::vector<char>& heavy,
                const std::vector<qsk::BatchState>& base, const std::vector<qsk::BatchOp>& ops) {
  P.L = L;
  P.cluster = cluster;
  P.states = base;
  std::vector<int> Ls(nq.size(), L);
  if (cluster > 1)
    for (size_t s = 0; s < nq.size(); ++s)
      if (heavy[s]) Ls[s] = std::min(L, nq[s] - (31 - __builtin_clz((unsigned)cluster)));
  qsbatch::build_segments(Ls, nq, P.states, ops, P.segs, P.xlat);
}

bool upload_plan(Plan& P) {
  const size_t S = P.states.size();
  if (qsalloc::device(reinterpret_cast<void**>(&P.d_states), sizeof(qsk::BatchState) * S) != cudaSuccess ||
      qsalloc::device(reinterpret_cast<void**>(&P.d_segs), sizeof(qsk::BatchSeg) * std::max<size_t>(1, P.segs.size())) != cudaSuccess ||
      qsalloc::device(reinterpret_cast<void**>(&P.d_xlat), sizeof(qsk::BatchXlat) * std::max<size_t>(1, P.xlat.size())) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (cudaMemcpy(P.d_states, P.states.data(), sizeof(qsk::BatchState) * S, cudaMemcpyHostToDevice) != cudaSuccess)
    return false;
  if (!P.segs.empty() && cudaMemcpy(P.d_segs, P.segs.data(), sizeof(qsk::BatchSeg) * P.segs.size(),
                                    cudaMemcpyHostToDevice) != cudaSuccess)
    return false;
  return P.xlat.empty() || cudaMemcpy(P.d_xlat, P.xlat.data(), sizeof(qsk::BatchXlat) * P.xlat.size(),
                                      cudaMemcpyHostToDevice) == cudaSuccess;
}

// Appends the packed tile passes of a state and where each starts (in units of 16
// bytes); nothing if it has an operation that does not fit.
void tile_passes(const qs_batch* b, int s, std::vector<unsigned char>* out, std::vector<uint32_t>* at) {
  const std::vector<qsk::BatchOp>& prog = b->progs[(size_t)s];
  std::vector<std::vector<int>> lists(3 * prog.size());     // controls, targets, Paulis
  std::vector<qstile::Gate> gates;
  for (size_t i = 0; i < prog.size(); ++i) {
    const qsk::BatchOp& op = prog[i];
    std::vector<int>&c = lists[3 * i], &t = lists[3 * i + 1], &pl = lists[3 * i + 2];
    const double* data = b->consts[(size_t)s].data() + op.coff;
    qstile::Gate g;
    g.kind = op.kind;
    if (op.kind == 2) {
      for (int q = 0; q < b->nq[(size_t)s]; ++q)
        if ((op.xy | op.yz) >> q & 1) {
          t.push_back(q);
          pl.push_back((op.xy >> q & 1) ? ((op.yz >> q & 1) ? 2 : 1) : 3);
        }
      g.c = data[0];
      g.s = data[1];
    } else {
      t.assign(op.t, op.t + op.n);
      for (int q = 0; q < b->nq[(size_t)s]; ++q)
        if (op.ctrl >> q & 1) c.push_back(q);
      g.data = data;
    }
    g.ctrls = &c;
    g.targs = &t;
    g.paulis = &pl;
    for (int q : c) g.qmask |= 1ull << q;
    for (int q : t) g.qmask |= 1ull << q;
    if (!qstile::fits(g, b->nq[(size_t)s])) return;
    gates.push_back(g);
  }
  qstile::build_passes(gates, b->nq[(size_t)s], [&](const qstile::TilePass& p) {
    at->push_back((uint32_t)(out->size() / 16));
    qstile::pack(p, out);
  });
}

// Two-qubit channels on the members of (t1, t2, t1 + N, t2 + N): member bits
// 0, 1 are t1, t2 and bits 2, 3 are t1 + N, t2 + N.
qs_status add_channel2(qs_batch* b, int state, int t1, int t2, bool depol, double p) {
  if (check_density(b, state) != QS_OK) return check_density(b, state);
  const int tt[2] = {t1, t2};
  qs_status st = qsapi::check_qubits(b->nlog[state], tt, 2, nullptr, 0);
  if (st != QS_OK) return st;
  return add_superop(b, state, {t1, t2}, qsbatch::channel2_superop(depol, p));
}

}  // namespace

extern "C" {

qs_status qs_batch_create(int num_states, const int* num_qubits, qs_prec prec, void* cuda_stream, qs_batch** out) {
  return qs_batch_create_mixed(num_states, num_qubits, nullptr, prec, cuda_stream, out);
}

qs_status qs_batch_create_mixed(int num_states, const int* num_qubits, const int* is_density, qs_prec prec,
                                void* cuda_stream, qs_batch** out) {
  if (!out || num_states < 1 || !num_qubits || (prec != QS_C64 && prec != QS_C128)) return QS_ERR_ARG;
  *out = nullptr;
  qs_batch* b = new (std::nothrow) qs_batch();
  if (!b) return QS_ERR_OOM;
  b->prec = prec;
  b->stream = static_cast<cudaStream_t>(cuda_stream);
  b->nlog.assign(num_qubits, num_qubits + num_states);
  b->dens.assign(num_states, 0);
  if (is_density)
    for (int s = 0; s < num_states; ++s) b->dens[s] = is_density[s] ? 1 : 0;
  for (int s = 0; s < num_states; ++s) b->nq.push_back(b->dens[s] ? 2 * b->nlog[s] : b->nlog[s]);
  b->progs.resize(num_states);
  b->consts.resize(num_states);
  size_t off = 0;
  for (int s = 0; s < num_states; ++s) {
    const int q = b->nq[s];
    if (b->nlog[s] < 1 || q > 24) {
      delete b;
      return QS_ERR_ARG;
    }
    b->offset.push_back(off);
    off += (size_t)1 << q;
    off = (off + 31) & ~(size_t)31;    // 256-byte aligned starts for complex64 and complex128
  }
  b->pool_amps = off;
  *out = b;
  return QS_OK;
}

qs_status qs_batch_destroy(qs_batch* b) {
  if (!b) return QS_ERR_ARG;
  free_device(b);
  if (b->capture_stream) cudaStreamDestroy(b->capture_stream);
  if (b->branch_stream) cudaStreamDestroy(b->branch_stream);
  delete b;
  return QS_OK;
}

qs_status qs_batch_pool_amps(const qs_batch* b, size_t* num_amps) {
  if (!b || !num_amps) return QS_ERR_ARG;
  *num_amps = b->pool_amps;
  return QS_OK;
}

qs_status qs_batch_state_offset(const qs_batch* b, int state, size_t* offset_amps) {
  if (check_state(b, state) != QS_OK || !offset_amps) return QS_ERR_ARG;
  *offset_amps = b->offset[state];
  return QS_OK;
}

qs_status qs_batch_bind_pool(qs_batch* b, void* d_pool) {
  if (!b || !d_pool) return QS_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(d_pool) % 256 != 0) return QS_ERR_ALIGN;
  b->pool = d_pool;
  b->compiled = false;
  return QS_OK;
}

qs_status qs_batch_add_unitary(qs_batch* b, int state, const int* ctrls, int nctrl, const int* targs, int ntarg,
                               const double* mat) {
  if (check_state(b, state) != QS_OK || !mat || ntarg < 1) return QS_ERR_ARG;
  if (ntarg > 2 || nctrl > 5) return QS_ERR_TOO_MANY_TARGETS;
  qs_status st = qsapi::check_qubits(b->nlog[state], targs, ntarg, ctrls, nctrl);
  if (st != QS_OK) return st;
  std::vector<int> c(ctrls, ctrls + nctrl), t(targs, targs + ntarg);
  st = add_dense(b, state, c, t, mat);
  if (st != QS_OK || !b->dens[state]) return st;
  // density matrix: U^* on t + N with controls c + N (Sec. "Unitary gates")
  const size_t nm = (size_t)2 << (2 * ntarg);
  std::vector<double> conj(mat, mat + nm);
  for (size_t i = 1; i < nm; i += 2) conj[i] = -conj[i];
  for (int& q : c) q += b->nlog[state];
  for (int& q : t) q += b->nlog[state];
  return add_dense(b, state, c, t, conj.data());
}

qs_status qs_batch_add_diagonal(qs_batch* b, int state, const int* targs, int ntarg, const double* diag) {
  if (check_state(b, state) != QS_OK || !diag || ntarg < 1) return QS_ERR_ARG;
  if (ntarg > 3) return QS_ERR_TOO_MANY_TARGETS;
  qs_status st = qsapi::check_qubits(b->nlog[state], targs, ntarg, nullptr, 0);
  if (st != QS_OK) return st;
  qsk::BatchOp op{};
  op.kind = 1;
  op.n = ntarg;
  for (int q = 0; q < ntarg; ++q) op.t[q] = targs[q];
  const size_t nd = (size_t)2 << ntarg;
  st = add(b, state, op, diag, nd);
  if (st != QS_OK || !b->dens[state]) return st;
  std::vector<double> conj(diag, diag + nd);   // density matrix: conj(d) on t + N
  for (size_t i = 1; i < nd; i += 2) conj[i] = -conj[i];
  for (int q = 0; q < ntarg; ++q) op.t[q] = targs[q] + b->nlog[state];
  return add(b, state, op, conj.data(), nd);
}

qs_status qs_batch_add_pauli_gadget(qs_batch* b, int state, const int* targs, const int* paulis, int n,
                                    double theta) {
  if (check_state(b, state) != QS_OK || n < 0 || (n > 0 && (!targs || !paulis))) return QS_ERR_ARG;
  qs_status st = qsapi::check_qubits(b->nlog[state], targs, n, nullptr, 0);
  if (st != QS_OK) return st;
  for (int q = 0; q < n; ++q)
    if (paulis[q] < 0 || paulis[q] > 3) return QS_ERR_ARG;
  auto one = [&](int shift, double th) {
    qsk::BatchOp op{};
    op.kind = 2;
    int ny = 0;
    for (int q = 0; q < n; ++q) {
      const int t = targs[q] + shift;
      if (paulis[q] == 1 || paulis[q] == 2) op.xy |= 1u << t;
      if (paulis[q] == 2 || paulis[q] == 3) op.yz |= 1u << t;
      if (paulis[q] == 2) ++ny;
    }
    op.eta = ny & 3;
    op.h = op.xy ? 31 - __builtin_clz(op.xy) : 0;
    const double phi = -0.5 * th;
    const double cs[2] = {std::cos(phi), std::sin(phi)};
    return add(b, state, op, cs, 2);
  };
  st = one(0, theta);
  if (st != QS_OK || !b->dens[state]) return st;
  int ny = 0;
  for (int q = 0; q < n; ++q) ny += paulis[q] == 2;
  // U(theta)^* = U((-1)^(#Y + 1) theta) on t + N (Algorithm "specific unitaries on density matrices")
  return one(b->nlog[state], (ny % 2 == 0) ? -theta : theta);
}

qs_status qs_batch_add_kraus(qs_batch* b, int state, const int* targs, int n, const double* kraus, int num_ops) {
  if (check_state(b, state) != QS_OK || !kraus || !targs || num_ops < 1 || n < 1) return QS_ERR_ARG;
  if (!b->dens[state]) return QS_ERR_NOT_DENSMATR;
  if (n > 2) return QS_ERR_TOO_MANY_TARGETS;
  qs_status st = qsapi::check_qubits(b->nlog[state], targs, n, nullptr, 0);
  if (st != QS_OK) return st;
  const std::vector<double> m = qsbatch::kraus_superop(n, kraus, num_ops);
  std::vector<int> t(targs, targs + n);
  for (int q = 0; q < n; ++q) t.push_back(targs[q] + b->nlog[state]);
  return add_dense(b, state, {}, t, m.data());
}

// The channels, in the paper's Choi-vector update rules (Sec. "Dephasing
// channel", "Depolarising channel", "Damping channel"), as superoperators.
qs_status qs_batch_add_dephasing(qs_batch* b, int state, int t, double p) {
  if (check_prob(p) != QS_OK) return QS_ERR_ARG;
  return add_channel1(b, state, t, 1.0, 0.0, 1.0 - 2.0 * p, 0.0);
}

qs_status qs_batch_add_depolarising(qs_batch* b, int state, int t, double p) {
  if (check_prob(p) != QS_OK) return QS_ERR_ARG;
  return add_channel1(b, state, t, 1.0 - 2.0 * p / 3.0, 2.0 * p / 3.0, 1.0 - 4.0 * p / 3.0, 0.0);
}

qs_status qs_batch_add_pauli_channel(qs_batch* b, int state, int t, double px, double py, double pz) {
  if (check_prob(px) != QS_OK || check_prob(py) != QS_OK || check_prob(pz) != QS_OK) return QS_ERR_ARG;
  return add_channel1(b, state, t, 1.0 - px - py, px + py, 1.0 - px - py - 2.0 * pz, px - py);
}

qs_status qs_batch_add_damping(qs_batch* b, int state, int t, double p) {
  if (check_prob(p) != QS_OK) return QS_ERR_ARG;
  if (check_density(b, state) != QS_OK) return check_density(b, state);
  qs_status st = qsapi::check_qubits(b->nlog[state], &t, 1, nullptr, 0);
  if (st != QS_OK) return st;
  return add_superop(b, state, {t}, qsbatch::damping_superop(p));
}

qs_status qs_batch_add_two_qubit_dephasing(qs_batch* b, int state, int t1, int t2, double p) {
  if (check_prob(p) != QS_OK) return QS_ERR_ARG;
  return add_channel2(b, state, t1, t2, false, p);
}

qs_status qs_batch_add_two_qubit_depolarising(qs_batch* b, int state, int t1, int t2, double p) {
  if (check_prob(p) != QS_OK) return QS_ERR_ARG;
  return add_channel2(b, state, t1, t2, true, p);
}

// with_passes: complex64 states whose operations fit may take tile passes.
static qs_status compile(qs_batch* b, int autotune, bool with_passes) {
  free_device(b);
  const int S = (int)b->nq.size();
  std::vector<qsk::BatchState> states(S);
  std::vector<qsk::BatchOp> ops;
  std::vector<double> consts;
  for (int s = 0; s < S; ++s) {
    states[s].offset = b->offset[s];
    states[s].nq = b->nq[s];
    states[s].first_op = (int)ops.size();
    states[s].nops = (int)b->progs[s].size();
    for (qsk::BatchOp op : b->progs[s]) {
      op.coff += consts.size();
      ops.push_back(op);
    }
    consts.insert(consts.end(), b->consts[s].begin(), b->consts[s].end());
  }
  b->total_ops = (long)ops.size();
  b->wide = 0;
  for (const auto& op : ops)
    if (op.kind == 0 && op.n > 2) b->wide = 1;
  const int sms = qsk::num_sms();
  // work per state; heavy: more than one CTA's share at two CTAs per SM
  std::vector<double> work(S);
  double total = 0.0;
  for (int s = 0; s < S; ++s) {
    double c = 1.0;
    for (const auto& op : b->progs[s]) c += qsbatch::op_cost(op);
    work[s] = c * (double)(1ull << b->nq[s]);
    total += work[s];
  }
  std::vector<char> heavy(S, 0);
  int nheavy = 0;
  for (int s = 0; s < S; ++s)
    if (b->nq[s] >= kHeavyMinQubits && work[s] > total / (2 * sms)) {
      heavy[s] = 1;
      ++nheavy;
    }
  // tile passes, level by level: pass k of every state that has one
  std::vector<char> tiled(S, 0);
  std::vector<unsigned char> passes;         // packed
  std::vector<qstile::TileItem> items;
  if (with_passes) {
    try {
      std::vector<std::vector<uint32_t>> of(S);   // where a state's passes start
      size_t levels = 0;
      for (int s = 0; s < S; ++s) {
        tile_passes(b, s, &passes, &of[s]);
        tiled[s] = !of[s].empty();
        levels = std::max(levels, of[s].size());
      }
      for (size_t k = 0; k < levels; ++k) {
        b->level.push_back((int)items.size());
        for (int s = 0; s < S; ++s)
          if (k < of[s].size())
            for (uint32_t t = 0; t < 1u << (b->nq[s] - qstile::kPassBits); ++t)
              items.push_back(qstile::TileItem{b->offset[s], of[s][k], t});
        if (items.size() > INT_MAX) throw std::bad_alloc();   // more than a launch numbers
      }
      b->level.push_back((int)items.size());
    } catch (const std::bad_alloc&) {             // without tile passes
      passes.clear();
      items.clear();
      b->level.clear();
      std::fill(tiled.begin(), tiled.end(), 0);
    }
  }
  // largest first, heavy ones before the others; a second list without the tiled states
  std::vector<int> order(S);
  for (int s = 0; s < S; ++s) order[s] = s;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    return heavy[x] != heavy[y] ? heavy[x] > heavy[y] : work[x] > work[y];
  });
  int rest = 0, rest_heavy = 0;
  for (int i = 0; i < S; ++i)
    if (const int s = order[i]; !tiled[s]) {
      order.push_back(s);
      ++rest;
      rest_heavy += heavy[s];
    }
  if (qsalloc::device(reinterpret_cast<void**>(&b->d_order), sizeof(int) * order.size()) != cudaSuccess ||
      (!passes.empty() &&
       (qsalloc::device(reinterpret_cast<void**>(&b->d_passes), passes.size()) != cudaSuccess ||
        qsalloc::device(reinterpret_cast<void**>(&b->d_items), sizeof(qstile::TileItem) * items.size()) != cudaSuccess)) ||
      qsalloc::device(reinterpret_cast<void**>(&b->d_ops), sizeof(qsk::BatchOp) * std::max<size_t>(1, ops.size())) != cudaSuccess ||
      qsalloc::device(reinterpret_cast<void**>(&b->d_consts), sizeof(double) * std::max<size_t>(1, consts.size())) != cudaSuccess ||
      qsalloc::device(reinterpret_cast<void**>(&b->d_counter), 2 * sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    free_device(b);
    return QS_ERR_OOM;
  }
  if (cudaMemcpy(b->d_order, order.data(), sizeof(int) * order.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      (!passes.empty() &&
       (cudaMemcpy(b->d_passes, passes.data(), passes.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->d_items, items.data(), sizeof(qstile::TileItem) * items.size(), cudaMemcpyHostToDevice) != cudaSuccess)) ||
      (!ops.empty() &&
       cudaMemcpy(b->d_ops, ops.data(), sizeof(qsk::BatchOp) * ops.size(), cudaMemcpyHostToDevice) != cudaSuccess) ||
      (!consts.empty() && cudaMemcpy(b->d_consts, consts.data(), sizeof(double) * consts.size(),
                                     cudaMemcpyHostToDevice) != cudaSuccess)) {
    free_device(b);
    return QS_ERR_CUDA;
  }
  // launch-shape candidates; each shared-memory size (tile size) has its own
  // segment plan, with and without heavy states shared by clusters
  if (qsk::batch_set_max_smem(200 * 1024) != cudaSuccess) {
    cudaGetLastError();
    return QS_ERR_CUDA;
  }
  struct Shape {
    int threads, per_sm, cluster;
    bool tiles;            // tile passes, and this launch for the rest
  };
  std::vector<Shape> cands;
  if (autotune) {
    cands = {{128, 4, 1, false}, {256, 2, 1, false}, {256, 4, 1, false}, {512, 1, 1, false}, {512, 2, 1, false}};
    // 512 complex64 states of 10-17 qubits: 1.54 ms without clusters, 1.22-1.38
    // in clusters of 2 and 4, 1.68 of 8; 256 complex128 states, a quarter of them
    // density matrices: 7.69, 3.75, 1.91 and 1.82 ms
    if (nheavy)
      cands.insert(cands.end(), {{512, 1, 2, false}, {512, 1, 4, false}, {256, 2, 4, false}, {256, 2, 8, false}});
    // tile passes: the 512 states in 0.61 ms
    if (!passes.empty()) cands.push_back({256, 2, rest_heavy ? 4 : 1, true});
  } else if (!passes.empty()) {
    cands = {{256, 2, rest_heavy ? 4 : 1, true}};
  } else {
    cands = {{256, 2, nheavy ? 4 : 1, false}};
  }
  std::vector<Plan> plans;
  plans.reserve(cands.size());       // pointers into it stay valid
  auto plan_for = [&](int L, int cluster) -> Plan* {
    for (auto& P : plans)
      if (P.L == L && P.cluster == cluster) return &P;
    plans.emplace_back();
    build_plan(plans.back(), L, cluster, b->nq, heavy, states, ops);
    return &plans.back();
  };
  for (const auto& c : cands) {
    Plan* P = plan_for(smem_qubits_for(b->prec, c.per_sm), c.cluster);
    if (!P->d_states && !upload_plan(*P)) {
      for (auto& Q : plans) Q.release();
      free_device(b);
      return QS_ERR_OOM;
    }
  }
  // the launches of a shape: the persistent one on st, the tile passes on tile_st
  auto launch = [&](const Plan& P, int threads, int ctas, int sq, int cluster, bool tiles, cudaStream_t st,
                    cudaStream_t tile_st) -> cudaError_t {
    cudaError_t e = cudaSuccess;
    const int n = tiles ? rest : S, nh = cluster > 1 ? (tiles ? rest_heavy : nheavy) : 0;
    if (n > 0) {
      e = cudaMemsetAsync(b->d_counter, 0, 2 * sizeof(int), st);
      if (e == cudaSuccess)
        e = qsk::launch_batch(b->prec, b->pool, P.d_states, b->d_order + (tiles ? S : 0), n, nh, b->d_ops, b->d_consts,
                              P.d_segs, P.d_xlat, b->d_counter, threads, ctas, sq, b->wide, cluster, st);
    }
    if (tiles)
      for (size_t k = 0; k + 1 < b->level.size() && e == cudaSuccess; ++k)
        e = qsk::launch_tile_items(b->pool, b->d_passes, b->d_items + b->level[k], b->level[k + 1] - b->level[k], tile_st);
    return e;
  };
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  float best = 1e30f;
  int best_plan = -1;
  bool best_tiles = false;
  for (const auto& c : cands) {
    const int sq = smem_qubits_for(b->prec, c.per_sm);
    Plan* P = plan_for(sq, c.cluster);
    int ctas = sms * c.per_sm;
    if (c.cluster > 1) {
      int n = 0;
      if (qsk::batch_max_clusters(b->prec, c.threads, sq, b->wide, c.cluster, &n) != cudaSuccess || n < 1) {
        cudaGetLastError();
        continue;
      }
      ctas = n * c.cluster;
    }
    cudaEventRecord(e0, b->stream);
    if (launch(*P, c.threads, ctas, sq, c.cluster, c.tiles, b->stream, b->stream) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaEventRecord(e1, b->stream);
    if (cudaEventSynchronize(e1) != cudaSuccess) return QS_ERR_CUDA;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best) {
      best = ms;
      b->threads = c.threads;
      b->ctas = ctas;
      b->smem_qubits = sq;
      b->cluster = c.cluster;
      best_tiles = c.tiles;
      best_plan = (int)(P - plans.data());
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  for (int i = 0; i < (int)plans.size(); ++i)
    if (i != best_plan) plans[i].release();
  if (b->ctas == 0 || best_plan < 0) return QS_ERR_CUDA;
  b->d_states = plans[best_plan].d_states;
  b->d_segs = plans[best_plan].d_segs;
  b->d_xlat = plans[best_plan].d_xlat;
  b->num_segs = (long)plans[best_plan].segs.size();
  b->best_ms = best;
  // record on the batch's own stream: reset the work counter, one persistent launch
  if (cudaStreamSynchronize(b->stream) != cudaSuccess) return QS_ERR_CUDA;
  for (cudaStream_t* st : {&b->capture_stream, &b->branch_stream})
    if (!*st && cudaStreamCreateWithFlags(st, cudaStreamNonBlocking) != cudaSuccess) return QS_ERR_CUDA;
  if (cudaStreamBeginCapture(b->capture_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return QS_ERR_CUDA;
  }
  // the persistent launch and the tile passes as two branches
  const Plan& P = plans[best_plan];
  const bool fork = best_tiles && rest > 0;
  cudaEvent_t forked = nullptr, joined = nullptr;
  cudaError_t e = cudaSuccess;
  if (fork) {
    e = cudaEventCreateWithFlags(&forked, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&joined, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(forked, b->capture_stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->branch_stream, forked, 0);
  }
  if (e == cudaSuccess)
    e = launch(P, b->threads, b->ctas, b->smem_qubits, b->cluster, best_tiles, b->capture_stream,
               fork ? b->branch_stream : b->capture_stream);
  if (fork && e == cudaSuccess) e = cudaEventRecord(joined, b->branch_stream);
  if (fork && e == cudaSuccess) e = cudaStreamWaitEvent(b->capture_stream, joined, 0);
  cudaGraph_t g = nullptr;
  const cudaError_t e2 = cudaStreamEndCapture(b->capture_stream, &g);
  if (forked) cudaEventDestroy(forked);
  if (joined) cudaEventDestroy(joined);
  if (e != cudaSuccess || e2 != cudaSuccess || !g) {
    cudaGetLastError();
    if (g) cudaGraphDestroy(g);
    return QS_ERR_CUDA;
  }
  b->graph = g;
  if (cudaGraphInstantiate(&b->exec, g, 0) != cudaSuccess) {
    cudaGetLastError();
    return QS_ERR_CUDA;
  }
  b->compiled = true;
  return QS_OK;
}

qs_status qs_batch_compile(qs_batch* b, int autotune) {
  if (!b || !b->pool) return QS_ERR_ARG;
  const bool c64 = b->prec == QS_C64;
  const qs_status st = compile(b, autotune, c64);
  // no device memory beside the tile passes' descriptors: the persistent launch alone
  return st == QS_ERR_OOM && c64 ? compile(b, autotune, false) : st;
}

qs_status qs_batch_run(qs_batch* b) {
  if (!b || !b->compiled) return QS_ERR_ARG;
  return cudaGraphLaunch(b->exec, b->stream) == cudaSuccess ? QS_OK : QS_ERR_CUDA;
}

qs_status qs_batch_info(const qs_batch* b, int* threads, int* ctas, int* smem_qubits, long* total_ops) {
  if (!b) return QS_ERR_ARG;
  if (threads) *threads = b->threads;
  if (ctas) *ctas = b->ctas;
  if (smem_qubits) *smem_qubits = b->smem_qubits;
  if (total_ops) *total_ops = b->total_ops;
  return QS_OK;
}

}  // extern "C"
