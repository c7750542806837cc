"""Batches whose largest states hold more than a CTA's share of the work, so that
the CTAs of a cluster share them: sizes from the least that is split up, states
that are all heavy, one heavy state among light ones, operations in global
memory between tiled ones, and density matrices, against the oracle."""

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# complex128 in double-float: about 2^-46 of the largest part per operation, 60
# operations twice; complex64: 2^-24 per operation likewise, amplitudes below 1
TOL = {1: 120 * 2.0 ** -46, 0: 120 * 2.0 ** -24}


@pytest.mark.parametrize("prec", [1, 0])
@pytest.mark.parametrize("autotune", [False, True])
@pytest.mark.parametrize("sizes,dens", [([11], []), ([12, 3], []), ([13, 13], []), ([15] + [4] * 20, []),
                                        ([10, 11, 12, 14, 16], []), ([6, 7, 5, 9], [0, 1])])
def test_heavy_states(sizes, dens, autotune, prec):
    import torch
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(len(sizes) + 10 * sizes[0])
    density = [s in dens for s in range(len(sizes))]
    batch = qs.Batch(sizes, prec=prec, density=density)
    circuits, inits = [], []
    for s, (nq, d) in enumerate(zip(sizes, density)):
        ops = (wl.small_densmatr_circuit if d else wl.unitary_circuit)(nq, 30, rng)
        if not d:
            ops.insert(10, {"op": "gadget", "targs": list(range(nq)), "paulis": [1 + q % 2 for q in range(nq)],
                            "theta": 0.7})           # flips every qubit: more than a tile pairs
            ops.insert(20, {"op": "diagonal", "targs": [nq - 1, 0], "diag": np.exp(1j * rng.uniform(0, 6, 4))})
        for op in ops:
            batch.add(s, op)
        circuits.append(ops)
        psi = wl.random_statevector(nq, rng)
        inits.append(orc.densmatr_from_pure(psi) if d else psi)
    batch.compile(autotune=autotune)
    for s, psi in enumerate(inits):
        batch.view(s).copy_(torch.from_numpy(psi.astype(np.complex128 if prec else np.complex64)))
    for _ in range(2):
        batch.run()
    torch.cuda.synchronize()
    for s, (psi, ops, d) in enumerate(zip(inits, circuits, density)):
        want = orc.run_ops(orc.run_ops(psi, ops, d), ops, d)
        assert np.max(np.abs(batch.view(s).cpu().numpy() - want)) <= TOL[prec], s


@pytest.mark.parametrize("nq,dens", [(12, False), (6, True)])
def test_segments_cost_no_bits(nq, dens):
    """A complex128 state gives the same bits whether it stays in shared memory (one of
    many) or is shared by a cluster, in small tiles that go through global memory between
    segments (alone, it is heavy).  (Gadgets that pair too many qubits for a small tile
    are left out: they run on the doubles in global memory.)"""
    import torch
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(5 + nq)
    ops = (wl.small_densmatr_circuit if dens else wl.unitary_circuit)(nq, 80, rng)
    ops = [op for op in ops if op["op"] != "gadget" or len(op["targs"]) <= 4]
    psi = wl.random_statevector(nq, rng)
    init = torch.from_numpy(orc.densmatr_from_pure(psi) if dens else psi)
    got = []
    for count in (1, 400):
        batch = qs.Batch([nq] * count, prec=qs.QS_C128, density=[dens] * count)
        for s in range(count):
            for op in ops:
                batch.add(s, op)
        batch.compile(autotune=False)
        for s in range(count):
            batch.view(s).copy_(init)
        batch.run()
        torch.cuda.synchronize()
        got.append(batch.view(0).cpu().numpy().copy())
    assert np.array_equal(got[0], got[1])
    want = orc.run_ops(init.numpy(), ops, is_density=dens)
    assert np.max(np.abs(got[0] - want)) <= len(ops) * 2.0 ** -46
