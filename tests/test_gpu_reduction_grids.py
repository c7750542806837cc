"""Norm, trace and Pauli sums at the sizes where their grids change: one block
(whose partial sum is the result), two blocks, the largest grids and the sizes
just above them, where a thread takes more than one item.  Against the oracle;
the bound is the FP64 sums' (2^-53 per addition of either side, at most
log2(n) + 30 deep here and in numpy's pairwise sums) relative to the sum of the
absolute values."""

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def tol(nq, prec_c64):
    return (2 * nq + 60) * 2.0 ** -53 + (2.0 ** -40 if prec_c64 else 0.0)


@pytest.mark.parametrize("c64", [False, True])
@pytest.mark.parametrize("nq", [1, 2, 5, 7, 8, 9, 10, 11, 18, 20, 21])
def test_statevector(nq, c64):
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(300 + nq)
    psi = wl.random_statevector(nq, rng)
    if c64:
        psi = psi.astype(np.complex64)
    wide = psi.astype(np.complex128)
    st = qs.State(nq, prec=qs.QS_C64 if c64 else qs.QS_C128)
    st.set_amps(psi)
    assert abs(qs.qs_calc_norm_or_trace(st.handle) - orc.calc_norm(wide)) <= tol(nq, c64)
    paulis, coeffs = wl.random_pauli_sum(nq, 6, rng)
    zs = np.where(rng.random((12, nq)) < 0.5, 3, 0).astype(np.int32)
    hz = rng.standard_normal(12)
    for p, h in ((paulis, coeffs), (zs, hz), (np.concatenate([paulis, zs]), np.concatenate([coeffs, hz]))):
        want = orc.expec_pauli_sum_statevector(wide, p, h)
        got = qs.qs_expec_pauli_sum(st.handle, p, h)
        assert abs(got - want) <= tol(nq, c64) * np.abs(h).sum()
        # the result of an earlier call leaves nothing behind
        assert abs(qs.qs_expec_pauli_sum(st.handle, p[:1], h[:1])
                   - orc.expec_pauli_sum_statevector(wide, p[:1], h[:1])) <= tol(nq, c64) * abs(h[0])
    st.close()


@pytest.mark.parametrize("c64", [False, True])
@pytest.mark.parametrize("nq,terms", [(1, 1), (1, 300), (3, 32), (3, 33), (6, 4), (6, 5), (8, 1), (9, 1), (10, 320)])
def test_density_matrix(nq, terms, c64):
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(400 + 10 * nq + terms)
    states, w = wl.random_mixed_state_vectors(nq, 3, rng)
    beta = sum(wi * orc.densmatr_from_pure(s) for wi, s in zip(w, states))
    if c64:
        beta = beta.astype(np.complex64)
    wide = beta.astype(np.complex128)
    dm = qs.State(nq, density=True, prec=qs.QS_C64 if c64 else qs.QS_C128)
    dm.set_amps(beta)
    assert abs(qs.qs_calc_norm_or_trace(dm.handle) - orc.calc_trace(wide)) <= tol(nq, False)
    paulis = rng.integers(0, 4, size=(terms, nq)).astype(np.int32)
    coeffs = rng.standard_normal(terms)
    want = orc.expec_pauli_sum_densmatr(wide, paulis, coeffs)
    assert abs(qs.qs_expec_pauli_sum(dm.handle, paulis, coeffs) - want) <= tol(nq + 9, False) * np.abs(coeffs).sum() * 2
    dm.close()
