"""Planned complex64 circuits in tile passes: from the smallest state that has a
tile (12 qubits) over sizes with few and many tiles, with every gate kind, controls
and diagonals inside and outside the tile, gadgets wider than a tile and dense gates
that do not fit (blocks between the runs), relabelled plans, and recorded programs.
Against the oracle in complex128.  The bound is on the 2-norm of the difference
relative to the state's: a two-target gate sums eight products (8 2^-24 and the
matrix's rounding, times at most 2 for the matrix of absolute values), so 20 2^-24 a
gate; tensor-core blocks keep to it too."""

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def circuit(nq, count, rng):
    ops = []
    for _ in range(count):
        q = [int(x) for x in rng.permutation(nq)]
        kind = int(rng.integers(0, 12))
        if kind < 3:
            nc = int(rng.integers(0, 4)) if kind else int(rng.integers(0, nq))
            ops.append({"op": "unitary", "ctrls": q[1:1 + nc], "targs": q[:1], "mat": wl.haar_unitary(2, rng)})
        elif kind < 5:
            nc = int(rng.integers(0, 4))
            ops.append({"op": "unitary", "ctrls": q[2:2 + nc], "targs": q[:2], "mat": wl.haar_unitary(4, rng)})
        elif kind < 7:
            n = int(rng.integers(1, 7))
            ops.append({"op": "diagonal", "targs": q[:n], "diag": np.exp(1j * rng.uniform(0, 6, 1 << n))})
        elif kind < 11:
            n = int(rng.integers(0, 7)) if kind < 10 else nq
            ops.append({"op": "gadget", "targs": q[:n], "paulis": [int(x) for x in rng.integers(0, 4, n)],
                        "theta": float(rng.uniform(0, 6))})
        else:
            ops.append({"op": "unitary", "ctrls": q[3:4], "targs": q[:3], "mat": wl.haar_unitary(8, rng)})
    return ops


@pytest.mark.parametrize("mode", ["plan", "relabel", "record"])
@pytest.mark.parametrize("nq", [11, 12, 13, 15, 19])
def test_circuits(nq, mode):
    import torch
    from paper_2311_01512_gb300 import costmodel, qs
    rng = np.random.default_rng(50 + nq)
    psi = wl.random_statevector(nq, rng)
    ops = circuit(nq, 70, rng)
    want = orc.run_ops(psi.astype(np.complex64).astype(np.complex128), ops, is_density=False)
    st = qs.State(nq, prec=qs.QS_C64, stream=torch.cuda.Stream())
    st.set_amps(psi)
    c = qs.Circuit(nq, ops)
    if mode == "relabel":
        model, _ = costmodel.load()
        c.plan_cost(model, st.handle, max_block_qubits=5, window=24)
        c.plan_relabel(model, st.handle, 7, 0.0)
        model.close()
    else:
        c.plan(qs.QS_PLAN_GREEDY, 4)
    if mode == "record":
        qs.qs_record_begin(st.handle)
        c.apply(st.handle)
        prog = qs.qs_record_end(st.handle)
        qs.qs_program_run(prog)
        qs.qs_synchronize(st.handle)
        got = st.get_amps()
        qs.qs_program_destroy(prog)
    else:
        c.apply(st.handle)
        qs.qs_synchronize(st.handle)
        got = st.get_amps()
    passes = qs.qs_test_circuit_passes(c)
    assert passes > 0 if nq >= 12 else passes == 0        # the runs were tile passes
    c.close()
    st.close()
    assert np.linalg.norm(got - want) <= (len(ops) + 1) * 20 * 2.0 ** -24 * np.linalg.norm(want)


def test_passes_are_formed_for_the_states_that_take_them():
    """A plan forms its tile passes when it first meets a complex64 statevector (of at
    least 12 qubits, with fused blocks), not for other states; and again for a new plan."""
    from paper_2311_01512_gb300 import costmodel, qs
    rng = np.random.default_rng(77)
    nq = 13
    ops = wl.unitary_circuit(nq, 60, rng)
    psi = wl.random_statevector(nq, rng)
    single, double = qs.State(nq, prec=qs.QS_C64), qs.State(nq)
    model, _ = costmodel.load()
    c = qs.Circuit(nq, ops)
    c.plan(qs.QS_PLAN_GREEDY, 4)
    double.set_amps(psi)
    c.apply(double.handle)
    assert qs.qs_test_circuit_passes(c) == -1
    single.set_amps(psi)
    c.apply(single.handle)
    assert qs.qs_test_circuit_passes(c) > 0
    c.plan_cost(model, double.handle, max_block_qubits=4, window=24)
    assert qs.qs_test_circuit_passes(c) == -1
    c.plan_cost(model, single.handle, max_block_qubits=4, window=24)
    assert qs.qs_test_circuit_passes(c) > 0
    c.plan(qs.QS_PLAN_NONE, 1)
    c.apply(single.handle)
    assert qs.qs_test_circuit_passes(c) == 0
    qs.qs_synchronize(single.handle)
    model.close()
    c.close()
    single.close()
    double.close()
