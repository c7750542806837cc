"""The measured workloads: what a user of this package has it do, through its
public entry points, from single calls on small states to circuits on
30-qubit ones.

A case fixes the shape of the work (sizes, operation kinds, qubits); the
amplitudes, gate matrices, angles, probabilities and coefficients come from
the seed.  Kinds of case:

* ``circuit``  operations applied one call each to a statevector;
* ``upload``   a state brought from page-locked host memory, a circuit, the norm;
* ``wide``     dense gates on a given number of targets, some controlled, one
               of them on the lowest qubits;
* ``density``  operations and channels applied one call each to a density
               matrix, then a partial trace, its trace and a Pauli sum;
* ``program``  the same operations recorded once and replayed;
* ``fused``    a circuit planned by the shipped cost model into fused blocks;
* ``batch``    many small states, each with its own circuit, in one launch;
* ``expect``   the expectation value of a Pauli sum on a statevector.
"""
import functools
import math

import numpy as np
import torch

from paper_2311_01512_gb300 import costmodel, qs
from paper_2311_01512_gb300 import workloads as wl

DEVICE = "cuda"


def listed():
    return [
        # a variational loop on a few qubits: every call is a launch on a 16 KiB state
        {"name": "circuit_10q", "kind": "circuit", "qubits": 10, "prec": "c128", "ops": 16, "circuit": 1},
        # a single-precision circuit on an odd, middling size, the state uploaded first
        {"name": "upload_25q_c64", "kind": "upload", "qubits": 25, "prec": "c64", "ops": 40, "circuit": 2},
        # the statevector benchmark's recipe and size
        {"name": "circuit_30q", "kind": "circuit", "qubits": 30, "prec": "c128", "ops": 40, "circuit": 3},
        # multi-target gates of a compiled circuit, two to five targets
        {"name": "wide_28q", "kind": "wide", "qubits": 28, "prec": "c128", "lo": 2, "hi": 5, "ops": 8, "circuit": 4},
        # the widest dense gate that the interface takes
        {"name": "wide6_25q", "kind": "wide", "qubits": 25, "prec": "c128", "lo": 6, "hi": 6, "ops": 2, "circuit": 5},
        # the 6-qubit noisy density-matrix workload, one call per operation
        {"name": "density_6q", "kind": "density", "qubits": 6, "recipe": "small", "ops": 60, "terms": 20,
         "trace": 2, "circuit": 6},
        # the same workload as a recorded program: what a parameter-free inner loop replays
        {"name": "program_6q", "kind": "program", "qubits": 6, "recipe": "small", "ops": 300, "circuit": 7},
        # a large noisy density matrix (28-qubit Choi vector)
        {"name": "density_14q", "kind": "density", "qubits": 14, "recipe": "large", "ops": 28, "terms": 100,
         "trace": 5, "circuit": 8},
        # a circuit known in advance, planned and fused, single precision
        {"name": "fused_29q_c64", "kind": "fused", "qubits": 29, "prec": "c64", "ops": 150, "block": 6,
         "circuit": 9},
        # a sweep of many small circuits, single precision
        {"name": "batch_c64", "kind": "batch", "prec": "c64", "states": 512, "lo": 10, "hi": 17, "density": 0,
         "ops": 60, "circuit": 10},
        # the same in double precision, one state in four a noisy density matrix
        {"name": "batch_c128", "kind": "batch", "prec": "c128", "states": 256, "lo": 10, "hi": 16, "density": 4,
         "ops": 60, "circuit": 11},
        # the energy of a Hamiltonian of local and long strings
        {"name": "expect_26q", "kind": "expect", "qubits": 26, "prec": "c128", "terms": 60, "circuit": 12},
    ]


def draw(rng):
    kind = rng.choice(["circuit", "circuit", "upload", "wide", "wide", "density", "density", "program", "fused",
                       "batch", "expect", "expect"])
    case = {"kind": kind, "circuit": rng.randrange(1, 1 << 20)}
    prec = rng.choice(["c128", "c128", "c64"])
    if kind == "circuit":
        case.update(qubits=rng.randint(7, 28), prec=prec, ops=rng.randint(8, 40))
    elif kind == "upload":
        case.update(qubits=rng.randint(12, 26), prec=prec, ops=rng.randint(4, 40))
    elif kind == "wide":
        n = rng.randint(2, 6)
        case.update(qubits=rng.randint(n + 4, 25 if n == 6 else 28), prec=prec, lo=n, hi=n, ops=rng.randint(2, 8))
    elif kind in ("density", "program"):
        small = kind == "program" or rng.random() < 0.5
        n = rng.randint(4, 8) if small else rng.randint(6, 13)
        case.update(qubits=n, recipe="small" if small else "large", ops=rng.randint(20, 60))
        if kind == "density":
            case.update(terms=rng.randint(1, 100), trace=rng.randint(1, n - 2))
    elif kind == "fused":
        case.update(qubits=rng.randint(20, 27), prec=prec, ops=rng.randint(50, 150), block=rng.randint(3, 5))
    elif kind == "batch":
        lo = rng.randint(7, 10)
        case.update(prec=prec, states=rng.randint(40, 256), lo=lo, hi=lo + rng.randint(1, 6),
                    density=rng.choice([0, 0, 3]), ops=rng.randint(20, 60))
    else:
        case.update(qubits=rng.randint(6, 26), prec=prec, terms=int(round(math.exp(rng.uniform(0, math.log(60))))))
    return case


# ---------------------------------------------------------------------------
# Operations: shapes from the case, values from the seed
# ---------------------------------------------------------------------------

def _wide_shapes(case, rng):
    """Dense gates on lo..hi targets, every width in turn: spread over all
    qubits with 0-2 controls, the last one uncontrolled on the lowest qubits."""
    n, ops = case["qubits"], []
    for k in range(case["ops"]):
        w = case["lo"] + k % (case["hi"] - case["lo"] + 1)
        c = min(int(rng.integers(0, 3)), n - w)
        q = [int(x) for x in rng.choice(n, size=w + c, replace=False)]
        if k == case["ops"] - 1:
            q, c = [int(x) for x in rng.permutation(w)], 0
        ops.append({"op": "unitary", "targs": q[:w], "ctrls": q[w:], "mat": np.empty((1 << w, 1 << w))})
    return ops


@functools.lru_cache(maxsize=64)
def _shapes(key):
    """The operations of a case with placeholder values (per state in a batch)."""
    case = dict(key)
    rng = np.random.default_rng([77, case["circuit"]])
    kind, n = case["kind"], case.get("qubits")
    if kind in ("circuit", "upload"):
        return wl.statevector_circuit(n, case["ops"], rng, max_targs=min(5, n - 1))
    if kind == "wide":
        return _wide_shapes(case, rng)
    if kind in ("density", "program"):
        recipe = wl.small_densmatr_circuit if case["recipe"] == "small" else wl.large_densmatr_circuit
        return recipe(n, case["ops"], rng)
    if kind == "fused":
        return wl.unitary_circuit(n, case["ops"], rng)
    sizes, dens, circs = [], [], []
    for s in range(case["states"]):
        d = bool(case["density"]) and s % case["density"] == 0
        q = int(rng.integers(case["lo"], case["hi"] + 1))
        q = max(3, q // 2) if d else q
        ops = int(rng.integers(case["ops"] // 2, case["ops"] + 1))
        sizes.append(q)
        dens.append(d)
        circs.append((wl.small_densmatr_circuit if d else wl.unitary_circuit)(q, ops, rng))
    return sizes, dens, circs


def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k != "name"))


class _Values:
    """Seeded values for operation shapes: Haar unitaries and channels from a
    pool per size, angles, phases and probabilities drawn one by one."""

    def __init__(self, seed):
        self.rng = np.random.default_rng([78, seed])
        self.pool = {}

    def pick(self, key, make):
        if key not in self.pool:
            self.pool[key] = [make() for _ in range(8)]
        return self.pool[key][int(self.rng.integers(8))]

    def fill(self, op):
        r, new = self.rng, dict(op)
        kind = op["op"]
        if kind == "unitary":
            d = 1 << len(op["targs"])
            new["mat"] = self.pick(("u", d), lambda: wl.haar_unitary(d, r))
        elif kind == "diagonal":
            new["diag"] = np.exp(1j * r.uniform(0.0, 2.0 * np.pi, size=1 << len(op["targs"])))
        elif kind == "gadget":
            new["theta"] = float(r.uniform(0.0, 2.0 * np.pi))
        elif kind == "kraus":
            q = len(op["targs"])
            new["kraus"] = self.pick(("k", q), lambda: wl.haar_kraus(q, 4, r))
        else:
            new["p"] = float(r.uniform(0.0, 0.1))
        return new


def _ops(case, seed):
    v = _Values(seed)
    return [v.fill(op) for op in _shapes(_key(case))]


def _hamiltonian(case, nq, seed):
    """Pauli strings (half of weight 1-4, half over all qubits) by the case,
    coefficients by the seed."""
    r = np.random.default_rng([79, case["circuit"]])
    p = np.zeros((case["terms"], nq), dtype=np.int32)
    for t in range(case["terms"]):
        if t % 2 == 0:
            targs, codes = wl.random_pauli_string(nq, 1, min(4, nq), r)
            p[t, targs] = codes
        else:
            p[t] = r.integers(0, 4, size=nq)
    return p, np.random.default_rng([80, seed]).standard_normal(case["terms"])


def _terms(case):
    return case.get("terms", 0)


# ---------------------------------------------------------------------------
# States
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(231101 + seed)
    return g


def _gaussian(n, seed, dtype=torch.complex128):
    """Normalised vector of complex Gaussian amplitudes."""
    v = torch.randn(1 << n, dtype=dtype, device=DEVICE, generator=_gen(seed))
    v /= torch.linalg.vector_norm(v)
    return v


def _mixture(n, seed):
    """Choi vector of a mixture of three Gaussian pure states."""
    w = np.random.default_rng([81, seed]).random(3)
    rho = torch.zeros(1 << (2 * n), dtype=torch.complex128, device=DEVICE)
    for k in range(3):
        psi = _gaussian(n, 16 * seed + k)
        m = rho.view(1 << n, 1 << n)          # [column, row]
        m += (w[k] / w.sum()) * psi.conj()[:, None] * psi[None, :]
    return rho


def _near_product(n, seed):
    """A product of random one-qubit states with some Gaussian noise on top:
    local expectation values of order one."""
    r = np.random.default_rng([82, seed])
    v = torch.ones(1, dtype=torch.complex128, device=DEVICE)
    for _ in range(n):
        q = r.standard_normal(2) + 1j * r.standard_normal(2)
        v = torch.kron(torch.tensor(q / np.linalg.norm(q), device=DEVICE), v)
    v += 0.3 * _gaussian(n, seed)
    v /= torch.linalg.vector_norm(v)
    return v


def _dtype(case):
    return torch.complex64 if case.get("prec") == "c64" else torch.complex128


def _prec(case):
    return qs.QS_C64 if case.get("prec") == "c64" else qs.QS_C128


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "batch":
        return _prepare_batch(case, seed, s)
    n = case["qubits"]
    if kind in ("density", "program"):
        stream = torch.cuda.Stream() if kind == "program" else None
        rho = _mixture(n, seed)
        if stream is not None:
            stream.wait_stream(torch.cuda.current_stream())
        s["state"] = qs.State(n, density=True, prec=qs.QS_C128, storage=rho, stream=stream)
        s["ops"] = _ops(case, seed)
        if kind == "density":
            s["paulis"], s["coeffs"] = _hamiltonian(case, n - case["trace"], seed)
        else:
            h = s["state"].handle
            qs.qs_record_begin(h)
            for op in s["ops"]:
                qs.apply_op(h, op)
            s["program"] = _Program(qs.qs_record_end(h), s["state"])
        return s
    if kind == "expect":
        s["state"] = qs.State(n, prec=_prec(case), storage=_near_product(n, seed).to(_dtype(case)))
        s["paulis"], s["coeffs"] = _hamiltonian(case, n, seed)
        return s
    psi = _gaussian(n, seed, _dtype(case))
    if kind == "upload":
        s["host"] = psi.cpu().pin_memory()
    s["state"] = qs.State(n, prec=_prec(case), storage=psi)
    s["ops"] = _ops(case, seed)
    if kind == "fused":
        model, _ = costmodel.load()
        s["circuit"] = qs.Circuit(n, s["ops"])
        s["circuit"].plan_cost(model, s["state"].handle, max_block_qubits=case["block"], window=24)
        model.close()
    return s


class _Program:
    """A recorded program, destroyed before its state."""

    def __init__(self, handle, state):
        self.handle, self.state = handle, state

    def __del__(self):
        try:
            qs.qs_program_destroy(self.handle)
        except Exception:
            pass


def _batch_members(case, seed):
    sizes, dens, circs = _shapes(_key(case))
    v = _Values(seed)
    return sizes, dens, [[v.fill(op) for op in c] for c in circs]


def _batch_amps(case, seed, sizes, dens, s):
    return _mixture(sizes[s], 997 * seed + s) if dens[s] else _gaussian(sizes[s], 997 * seed + s, _dtype(case))


def _prepare_batch(case, seed, s):
    sizes, dens, circs = _batch_members(case, seed)
    b = qs.Batch(sizes, prec=_prec(case), density=dens)
    for k, c in enumerate(circs):
        for op in c:
            b.add(k, op)
    b.compile(autotune=True)
    b.pool.zero_()
    for k in range(len(sizes)):
        b.view(k).copy_(_batch_amps(case, seed, sizes, dens, k))
    s["batch"] = b
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        s["batch"].run()
        return s["batch"].pool
    st = s["state"]
    h = st.handle
    if kind == "program":
        qs.qs_program_run(s["program"].handle)
        return st.tensor
    if kind == "expect":
        return np.float64(qs.qs_expec_pauli_sum(h, s["paulis"], s["coeffs"]).real)
    if kind == "fused":
        s["circuit"].apply(h)
        return st.tensor
    if kind == "upload":
        qs.qs_set_amps_ptr(h, s["host"].data_ptr(), 0, s["host"].numel())
    for op in s["ops"]:
        qs.apply_op(h, op)
    if kind == "upload":
        return st.tensor, np.float64(qs.qs_calc_norm_or_trace(h).real)
    if kind == "density":
        red = st.partial_trace(list(range(s["case"]["trace"])))
        tr = qs.qs_calc_norm_or_trace(red.handle)
        e = qs.qs_expec_pauli_sum(red.handle, s["paulis"], s["coeffs"])
        out = (st.tensor, red.tensor, np.float64(tr.real), np.float64(e.real))
        red.close()
        return out
    return st.tensor


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

def _op_work(op, n, density):
    """(share of the state's amplitudes that the operation changes, flops per
    changed amplitude)."""
    kind = op["op"]
    if kind == "unitary":
        f = 0.5 ** len(op["ctrls"])
        return (f if not density else 2 * f - f * f), 8.0 * (1 << len(op["targs"])) * (2 if density else 1)
    if kind == "diagonal":
        return 1.0, 6.0 * (2 if density else 1)
    if kind == "gadget":
        return 1.0, 8.0 * (2 if density else 1)
    if kind == "kraus":
        return 1.0, 8.0 * 16
    return {"dephasing": (0.5, 2.0), "dephasing2": (0.75, 2.0), "depolarising": (1.0, 4.0),
            "depolarising2": (1.0, 4.0), "damping": (1.0, 3.0)}[kind]


def _circuit_work(ops, n, size, density, one_pass):
    """One read and one write of what each call changes, or of the state once
    where the whole circuit is in hand."""
    amps = float(1 << (2 * n if density else n))
    w = [_op_work(op, n, density) for op in ops]
    return 2 * size * amps * (1.0 if one_pass else sum(f for f, _ in w)), amps * sum(f * k for f, k in w)


def work(case):
    kind = case["kind"]
    size = 8 if case.get("prec") == "c64" else 16
    if kind == "batch":
        sizes, dens, circs = _shapes(_key(case))
        w = [_circuit_work(c, q, size, d, True) for q, d, c in zip(sizes, dens, circs)]
        return {"bytes": sum(x for x, _ in w), "flops": sum(x for _, x in w)}
    n = case["qubits"]
    if kind == "expect":
        p, _ = _hamiltonian(case, n, 0)
        diag = sum(1 for t in p if not np.any((t == 1) | (t == 2)))
        return {"bytes": float(size << n), "flops": float(1 << n) * (2.0 * (case["terms"] - diag) + 3.0)}
    density = kind in ("density", "program")
    b, f = _circuit_work(_shapes(_key(case)), n, size, density, kind in ("program", "fused"))
    if kind == "upload":
        b += 3.0 * (size << n)                # the host buffer read, the state written, and read for its norm
        f += 4.0 * (1 << n)
    if kind == "density":
        left = n - case["trace"]
        b += 16.0 * ((1 << (2 * n - case["trace"])) + (1 << (2 * left)))
        b += 16.0 * (1 << left) * (1 + case["terms"])
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the difference from 64-bit sums that was measured: one
    rounding per operation in double precision (47-bit arithmetic in
    double-precision batches); single-precision operations, and for fused
    blocks the tensor cores' single-precision accumulation.  A Pauli sum
    cancels, so its rounding is relative to a value below that of its terms."""
    kind, single = case["kind"], case.get("prec") == "c64"
    if kind == "expect":
        return {"rel": 4e-6 if single else 1e-13}
    if single:
        return {"rel": {"fused": 3e-5, "batch": 2e-6}.get(kind, 6e-6)}
    return {"rel": 2e-13 if kind == "batch" else 8e-15}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _dense64(v, n, targs, ctrls, mat):
    """mat on the target bits of v's indices (matrix bit q on targs[q]) where
    every control bit is 1, in place."""
    pos = sorted(targs + ctrls, reverse=True)
    shape, axis, top = [], {}, n
    for p in pos:
        shape += [1 << (top - 1 - p), 2]
        axis[p] = len(shape) - 1
        top = p
    sub = v.view(shape + [1 << top])
    for c in sorted(ctrls):                   # ascending position: descending axis
        sub = sub.select(axis[c], 1)
        for p in axis:
            axis[p] -= axis[p] > axis[c]
    order = [axis[t] for t in reversed(targs)]
    sub = sub.permute(order + [a for a in range(sub.dim()) if a not in order])
    m = torch.as_tensor(np.ascontiguousarray(mat, dtype=np.complex128), device=v.device)
    sub.copy_((m @ sub.reshape(m.shape[0], -1)).view(sub.shape))


def _parity(x):
    for k in (32, 16, 8, 4, 2, 1):
        x = x ^ (x >> k)
    return (x & 1).to(torch.float64)


def _string(targs, paulis):
    xy = sum(1 << t for t, p in zip(targs, paulis) if p in (1, 2))
    yz = sum(1 << t for t, p in zip(targs, paulis) if p in (2, 3))
    return xy, yz, 1j ** (sum(1 for p in paulis if p == 2) % 4)


def _pauli64(v, i, xy, yz, eta):
    """(P v)_i for a Pauli string P."""
    j = i ^ xy
    return (eta * (1.0 - 2.0 * _parity(j & yz))) * v[j]


def _chunks(n):
    step = 1 << min(n, 25)
    for b in range(0, 1 << n, step):
        yield torch.arange(b, b + step, device=DEVICE)


def _gadget64(v, n, targs, paulis, theta):
    xy, yz, eta = _string(targs, paulis)
    new = torch.empty_like(v)
    for i in _chunks(n):
        lo = int(i[0])
        new[lo:lo + i.numel()] = math.cos(theta / 2) * v[i] - 1j * math.sin(theta / 2) * _pauli64(v, i, xy, yz, eta)
    v.copy_(new)


def _channel64(op):
    """Superoperator of a channel as sum conj(K) (x) K."""
    kind, p = op["op"], op.get("p", 0.0)
    x = [np.eye(2), np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.diag([1, -1])]
    if kind == "kraus":
        ks = op["kraus"]
    elif kind == "dephasing":
        ks = [math.sqrt(1 - p) * x[0], math.sqrt(p) * x[3]]
    elif kind == "depolarising":
        ks = [math.sqrt(1 - p) * x[0]] + [math.sqrt(p / 3) * x[k] for k in (1, 2, 3)]
    elif kind == "damping":
        ks = [np.diag([1.0, math.sqrt(1 - p)]), np.array([[0, math.sqrt(p)], [0, 0]])]
    elif kind == "dephasing2":
        ks = [math.sqrt(1 - p) * np.eye(4)] + [math.sqrt(p / 3) * np.kron(x[a], x[b])
                                               for a, b in ((0, 3), (3, 0), (3, 3))]
    else:
        ks = [math.sqrt(1 - p) * np.eye(4)] + [math.sqrt(p / 15) * np.kron(x[a], x[b])
                                               for a in range(4) for b in range(4) if a + b]
    return sum(np.kron(np.conj(k), k) for k in ks)


def _apply64(v, n, op, density):
    kind = op["op"]
    full = 2 * n if density else n
    if kind in ("unitary", "diagonal"):
        m = np.asarray(op["mat"] if kind == "unitary" else np.diag(op["diag"]))
        c = list(op.get("ctrls", []))
        _dense64(v, full, list(op["targs"]), c, m)
        if density:
            _dense64(v, full, [t + n for t in op["targs"]], [t + n for t in c], m.conj())
    elif kind == "gadget":
        _gadget64(v, full, op["targs"], op["paulis"], op["theta"])
        if density:
            flip = 1 if sum(1 for p in op["paulis"] if p == 2) % 2 else -1
            _gadget64(v, full, [t + n for t in op["targs"]], op["paulis"], flip * op["theta"])
    else:
        t = list(op["targs"])
        _dense64(v, full, t + [q + n for q in t], [], _channel64(op))


def _expect64(v, n, paulis, coeffs):
    total = 0.0
    for row, h in zip(paulis, coeffs):
        xy, yz, eta = _string(range(n), [int(c) for c in row])
        part = [torch.sum(v[i].conj() * _pauli64(v, i, xy, yz, eta)).real for i in _chunks(n)]
        total += float(h) * float(torch.stack(part).sum())
    return total


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sizes, dens, circs = _batch_members(case, seed)
        out, off = [], 0
        for k, (q, d, c) in enumerate(zip(sizes, dens, circs)):
            v = _batch_amps(case, seed, sizes, dens, k).to(torch.complex128)
            for op in c:
                _apply64(v, q, op, d)
            out.append(v)
            pad = -(off + v.numel()) % 32     # every state starts on a multiple of 32 amplitudes
            out.append(torch.zeros(pad, dtype=v.dtype, device=v.device))
            off += v.numel() + pad
        return torch.cat(out)
    n = case["qubits"]
    if kind == "expect":
        v = _near_product(n, seed).to(_dtype(case)).to(torch.complex128)
        return np.float64(_expect64(v, n, *_hamiltonian(case, n, seed)))
    density = kind in ("density", "program")
    v = _mixture(n, seed) if density else _gaussian(n, seed, _dtype(case)).to(torch.complex128)
    for op in _ops(case, seed):
        _apply64(v, n, op, density)
    if kind == "upload":
        return v, np.float64(float(torch.sum(torch.view_as_real(v).square())))
    if kind == "density":
        k = case["trace"]
        m = v.view(1 << (n - k), 1 << k, 1 << (n - k), 1 << k)
        red = torch.einsum("cvrv->cr", m).contiguous()
        e = 0.0
        dim = 1 << (n - k)
        r = torch.arange(dim, device=DEVICE)
        p, h = _hamiltonian(case, n - k, seed)
        for row, w in zip(p, h):              # Tr(P rho) = sum_r P[r, c] rho[c, r]: P rho's diagonal
            xy, yz, eta = _string(range(n - k), [int(c) for c in row])
            j = r ^ xy
            e += float(w) * float(torch.sum(eta * (1.0 - 2.0 * _parity(j & yz)) * red[r, j]).real)
        return v, red.reshape(-1), np.float64(float(torch.sum(torch.diagonal(red)).real)), np.float64(e)
    return v
