"""complex64 batches in tile passes: states of one tile and of many, states with
different numbers of passes and none, density matrices whose operations all fit,
and smaller states run beside them; twice in a row, against the oracle."""

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,dens", [([12], []), ([12, 13, 16, 14, 13], []), ([15, 3, 12, 11, 8, 12], []),
                                        ([6, 7, 13, 5], [0, 1, 3])])
def test_tiled_states(sizes, dens):
    import torch
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(17 + sum(sizes))
    density = [s in dens for s in range(len(sizes))]
    batch = qs.Batch(sizes, prec=qs.QS_C64, density=density)
    circuits, inits = [], []
    for s, (nq, d) in enumerate(zip(sizes, density)):
        ops = wl.unitary_circuit(nq, 0 if s == 4 else 15 * (s + 1), rng)
        for k in range(4):
            n = min(nq, 3)
            ops.insert(min(len(ops), 5 * k), {"op": "diagonal", "targs": [int(q) for q in rng.permutation(nq)[:n]],
                                              "diag": np.exp(1j * rng.uniform(0, 6, 1 << n))})
            if d:
                ops.insert(3, {"op": "damping", "targs": [k], "p": 0.1})
                ops.insert(9, {"op": "depolarising", "targs": [nq - 1 - k], "p": 0.05})
        if s == 4:
            ops = []
        for op in ops:
            batch.add(s, op)
        circuits.append(ops)
        psi = wl.random_statevector(nq, rng)
        inits.append(orc.densmatr_from_pure(psi) if d else psi)
    batch.compile(autotune=False)
    for s, psi in enumerate(inits):
        batch.view(s).copy_(torch.from_numpy(psi.astype(np.complex64)))
    for _ in range(2):
        batch.run()
    torch.cuda.synchronize()
    for s, (psi, ops, d) in enumerate(zip(inits, circuits, density)):
        want = orc.run_ops(orc.run_ops(psi, ops, d), ops, d)
        # 20 2^-24 of the norm a gate (a density matrix's gates are two operations each)
        bound = (2 * len(ops) * (2 if d else 1) + 1) * 20 * 2.0 ** -24 * max(1.0, np.linalg.norm(want))
        assert np.linalg.norm(batch.view(s).cpu().numpy() - want) <= bound, s


@pytest.mark.parametrize("autotune", [False, True])
def test_without_memory_for_the_passes(autotune):
    """A batch whose descriptors do not fit into device memory beside those of its tile
    passes, whichever allocation finds that out, runs in the persistent launch alone; if
    that does not fit either, it is reported and the batch compiles afterwards."""
    import torch
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(31)
    sizes = [13, 12, 9]
    batch = qs.Batch(sizes, prec=qs.QS_C64)
    circuits = [wl.unitary_circuit(nq, 20, rng) for nq in sizes]
    for s, ops in enumerate(circuits):
        for op in ops:
            batch.add(s, op)
    inits = [wl.random_statevector(nq, rng) for nq in sizes]
    for skip in range(8):
        try:
            qs.qs_test_fail_allocations(skip, 1)
            batch.compile(autotune=autotune)
        finally:
            qs.qs_test_fail_allocations(0, 0)
        for s, psi in enumerate(inits):
            batch.view(s).copy_(torch.from_numpy(psi.astype(np.complex64)))
        batch.run()
        torch.cuda.synchronize()
        for s, (psi, ops) in enumerate(zip(inits, circuits)):
            want = orc.run_ops(psi, ops, is_density=False)
            assert np.linalg.norm(batch.view(s).cpu().numpy() - want) <= (len(ops) + 1) * 20 * 2.0 ** -24, (skip, s)
    try:
        qs.qs_test_fail_allocations(0, 100)
        with pytest.raises(qs.QSError) as ei:
            batch.compile(autotune=autotune)
        assert "QS_ERR_OOM" in str(ei.value)
    finally:
        qs.qs_test_fail_allocations(0, 0)
    batch.compile(autotune=autotune)
