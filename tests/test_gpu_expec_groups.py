"""Statevector expectation values whose terms share flip masks in runs of every
length around the kernels' switch from per-term products to a product formed
once per element, on states around one 1024-amplitude tile."""

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# Rounding of a sum of 2^nq products per term, per unit of sum |h| (the state is
# normalised): FP64 below 2^-46 for nq <= 12; double-float and complex64 parts
# (47-bit and 24-bit inputs) as the other expectation tests take them.
TOL = {"fx": 1.4e-14, "df": 1e-12, "c64": 1e-5}


@pytest.mark.parametrize("mode", ["fx", "df", "c64"])
@pytest.mark.parametrize("nq", [1, 3, 9, 10, 11, 12])
def test_groups_of_shared_masks(mode, nq):
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(640 + nq)
    psi = wl.random_statevector(nq, rng)
    st = qs.State(nq, prec=qs.QS_C64 if mode == "c64" else qs.QS_C128)
    if mode == "df":
        qs.qs_set_arithmetic(st.handle, qs.QS_ARITH_DF)
    st.set_amps(psi)
    if mode == "c64":
        psi = psi.astype(np.complex64).astype(np.complex128)
    rows = []
    for count in (1, 2, 4, 5, 7):                      # terms per mask
        base = rng.integers(0, 4, size=nq)
        base[rng.integers(nq)] = 1                      # at least one flip
        for _ in range(count):
            flips = (base == 1) | (base == 2)           # same mask, every number of Y mod 4 turns up
            rows.append(np.where(flips, rng.choice([1, 2], size=nq), rng.choice([0, 3], size=nq)))
    for q in {0, min(4, nq - 1), min(8, nq - 1), nq - 1}:   # highest flip bit in a warp, an element, a tile
        rows.append(np.where(np.arange(nq) == q, 2, 3))
    paulis = np.array(rows, dtype=np.int32)
    coeffs = rng.standard_normal(len(rows))
    got = qs.qs_expec_pauli_sum(st.handle, paulis, coeffs)
    want = orc.expec_pauli_sum_statevector(psi, paulis, coeffs)
    st.close()
    assert got.imag == 0.0
    assert abs(got - want) < TOL[mode] * np.abs(coeffs).sum()
