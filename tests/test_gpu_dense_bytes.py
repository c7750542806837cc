"""Complex128 dense gates on the byte-sliced tensor-core kernels at the edges of
their tiles: fewer groups than a tile's 128 rows, passes of fewer tiles than SMs and of
many per CTA (the rings' phases go round several times), controls, amplitudes and matrices of widely
spread magnitudes, and the conjugate and superoperator passes of density
matrices.  Against the oracle within the kernels' error bound."""

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def bound(n, amps, mat):
    """Per output: 2^-55 of the row's largest per amplitude (K real terms), half
    a unit of the recombined sum and the dropped products (together below
    2^-52), in units of the largest amplitude times the largest entry; one final
    rounding; and the oracle's own K-term FP64 sum (K 2^-53)."""
    K = 2 << n
    return (K / 8 + 2 + K / 2) * 2.0 ** -52 * np.abs(amps.view(np.float64)).max() * np.abs(np.asarray(mat).view(np.float64)).max()


@pytest.mark.parametrize("spread", [0, 40])
@pytest.mark.parametrize("n,nq", [(3, 3), (3, 9), (3, 18), (3, 22), (4, 5), (4, 12), (4, 19), (4, 22), (5, 5), (5, 8), (5, 12), (5, 19),
                                  (5, 23), (6, 6), (6, 7), (6, 12), (6, 13), (6, 14), (6, 20), (6, 23)])
def test_dense_gate(n, nq, spread):
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(6400 + 100 * n + nq)
    psi = wl.random_statevector(nq, rng)
    mat = np.ascontiguousarray(wl.haar_unitary(1 << n, rng))
    if spread:                                  # magnitudes over 40 binades, exact zeros among them
        psi *= 2.0 ** -rng.integers(0, spread, size=psi.size)
        psi[rng.integers(0, psi.size, size=max(1, psi.size // 8))] = 0.0
        mat = mat * 2.0 ** -rng.integers(0, spread, size=mat.shape)
    for targs, ctrls in ((list(rng.permutation(nq)[:n]), []), (list(range(n)), []),
                         (list(rng.permutation(nq)[:n]), None)):
        targs = [int(t) for t in targs]
        if ctrls is None:
            ctrls = [q for q in range(nq) if q not in targs][:2]
        st = qs.State(nq)
        st.set_amps(psi)
        qs.qs_apply_ctrl_multi_target(st.handle, ctrls, targs, mat)
        qs.qs_synchronize(st.handle)
        got = st.get_amps()
        st.close()
        want = orc.run_ops(psi, [{"op": "unitary", "ctrls": ctrls, "targs": targs, "mat": mat}], is_density=False)
        assert np.max(np.abs((got - want).view(np.float64))) <= bound(n, psi, mat)


@pytest.mark.parametrize("n", [2, 3, 4, 5])
@pytest.mark.parametrize("extra", [0, 1, 2, 5, 8, 11, 12, 13, 14])
def test_small_passes(n, extra):
    """Dense blocks and gates with controls around the size where passes change
    from one thread per amplitude to the tensor cores."""
    from paper_2311_01512_gb300 import qs
    nq = n + extra
    rng = np.random.default_rng(700 + 20 * n + extra)
    psi = wl.random_statevector(nq, rng) * 2.0 ** -rng.integers(0, 12, size=1 << nq)
    mat = np.ascontiguousarray(wl.haar_unitary(1 << n, rng))
    perm = [int(q) for q in rng.permutation(nq)]
    for ctrls in ([], perm[n:n + 1], perm[n:n + 3]):
        st = qs.State(nq)
        st.set_amps(psi)
        if ctrls:
            qs.qs_apply_ctrl_multi_target(st.handle, ctrls, perm[:n], mat)
        else:
            qs.qs_apply_dense_block(st.handle, perm[:n], mat)
        got = st.get_amps()
        st.close()
        want = orc.run_ops(psi, [{"op": "unitary", "ctrls": ctrls, "targs": perm[:n], "mat": mat}], is_density=False)
        assert np.max(np.abs((got - want).view(np.float64))) <= bound(n, psi, mat)


def test_repeated_gates_share_the_scratch():
    """Six-target gates with different matrices queued back to back, and through
    a recorded program replayed twice."""
    import torch
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(66)
    nq = 14
    psi = wl.random_statevector(nq, rng)
    ops = [{"op": "unitary", "ctrls": [], "targs": [int(t) for t in rng.permutation(nq)[:6]],
            "mat": wl.haar_unitary(64, rng)} for _ in range(5)]
    stream = torch.cuda.Stream()
    st = qs.State(nq, stream=stream)
    st.set_amps(psi)
    for op in ops:
        qs.apply_op(st.handle, op)
    want = orc.run_ops(psi, ops, is_density=False)
    assert np.max(np.abs(st.get_amps() - want)) < 1e-14
    qs.qs_record_begin(st.handle)
    for op in ops:
        qs.apply_op(st.handle, op)
    prog = qs.qs_record_end(st.handle)
    for _ in range(2):
        qs.qs_program_run(prog)
        want = orc.run_ops(want, ops, is_density=False)
    assert np.max(np.abs(st.get_amps() - want)) < 1e-14
    qs.qs_program_destroy(prog)
    st.close()


@pytest.mark.parametrize("nq", [4, 8, 9])
def test_density_matrix_passes(nq):
    """Three-qubit Kraus maps (a six-target superoperator), two-qubit ones,
    and the two passes of
    controlled and wide unitaries."""
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(67 + nq)
    rho = orc.densmatr_from_pure(wl.random_statevector(nq, rng))
    ops = [{"op": "kraus", "targs": [3, 0, 2], "kraus": wl.haar_kraus(3, 3, rng)},
           {"op": "kraus", "targs": [2, 0], "kraus": wl.haar_kraus(2, 4, rng)},
           {"op": "unitary", "ctrls": [], "targs": [3, 1], "mat": wl.haar_unitary(4, rng)},
           {"op": "unitary", "ctrls": [], "targs": [2, 0, 3, 1], "mat": wl.haar_unitary(16, rng)},
           {"op": "unitary", "ctrls": [1], "targs": [2, 0, 3], "mat": wl.haar_unitary(8, rng)}]
    st = qs.State(nq, density=True)
    st.set_amps(rho)
    for op in ops:
        qs.apply_op(st.handle, op)
    got = st.get_amps()
    st.close()
    assert np.max(np.abs(got - orc.run_ops(rho, ops, is_density=True))) < 1e-14


@pytest.mark.parametrize("arith", ["fx", "df"])
@pytest.mark.parametrize("nq", [2, 4, 7, 8])
def test_two_qubit_superoperator_host_and_device(nq, arith):
    """Kraus maps of at most 16 operators on small states have their superoperator
    formed on the host, the same map with zero operators appended on the device:
    the same operations, hence equal results; and the map against the oracle."""
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(1600 + nq)
    states, w = wl.random_mixed_state_vectors(nq, 3, rng)
    beta = sum(wi * orc.densmatr_from_pure(s) for wi, s in zip(w, states))
    for m in (1, 4, 16):
        kraus = list(wl.haar_kraus(2, m, rng))
        zeros = [np.zeros((4, 4), dtype=np.complex128)] * (17 - m)
        t = [int(q) for q in rng.permutation(nq)[:2]]
        got = []
        for ops in (kraus, kraus + zeros):
            dm = qs.State(nq, density=True, prec=qs.QS_C128)
            qs.qs_set_arithmetic(dm.handle, qs.QS_ARITH_FX if arith == "fx" else qs.QS_ARITH_DF)
            dm.set_amps(beta)
            qs.qs_apply_kraus(dm.handle, t, ops)
            got.append(dm.get_amps())
            dm.close()
        assert np.array_equal(got[0], got[1])
        want = orc.densmatr_apply_kraus(beta, t, kraus)
        assert np.max(np.abs((got[0] - want).view(np.float64))) <= bound(4, beta, orc.superoperator(kraus))
