"""Complex128 dense gates whose results leave the normal numbers: below 2^-1022 they
become subnormal numbers or zero and above 2^1024 infinities, as in FP64, in every row
of a tile and beside rows of zeros.  The reference is the oracle at exponent 0 (the
gate is linear), scaled afterwards."""

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def scaled(v, e):
    p = v.view(np.float64)
    return np.ldexp(np.ldexp(p, e // 2), e - e // 2).view(np.complex128)


def apply(nq, density, targs, mat, psi):
    from paper_2311_01512_gb300 import qs
    st = qs.State(nq, density=density)
    st.set_amps(psi)
    qs.qs_apply_ctrl_multi_target(st.handle, [], targs, mat)
    qs.qs_synchronize(st.handle)
    got = st.get_amps()
    st.close()
    return got


@pytest.mark.parametrize("e_amp,e_mat", [(-980, -20), (-950, -60), (-1000, 0), (-500, -500)])
@pytest.mark.parametrize("n,nq,density", [(3, 8, False), (3, 20, False), (4, 18, False), (5, 18, False), (6, 9, False),
                                          (3, 5, True), (4, 5, True)])
def test_small_results(n, nq, density, e_amp, e_mat):
    """Amplitudes over 30 binades, so that results lie on both sides of 2^-1022."""
    rng = np.random.default_rng(90 + 10 * n + nq)
    size = 1 << (2 * nq if density else nq)
    psi = (rng.standard_normal(size) + 1j * rng.standard_normal(size)) * 2.0 ** -rng.integers(0, 30, size=size)
    psi[: size // 2] *= 2.0 ** -20
    psi[rng.integers(0, size, size=size // 8)] = 0.0
    mat = wl.haar_unitary(1 << n, rng)
    targs = [int(t) for t in rng.permutation(nq)[:n]]
    want = orc.run_ops(psi, [{"op": "unitary", "ctrls": [], "targs": targs, "mat": mat}], is_density=density)
    passes = 2 if density else 1
    got = apply(nq, density, targs, scaled(mat, e_mat), scaled(psi, e_amp))
    e = e_amp + passes * e_mat
    K = 2 << n
    # per pass the kernels' bound (K 2^-55 of the group's largest amplitude and the oracle's
    # own K 2^-53), the flush of inputs and outputs below the smallest normal number
    tol = passes * K * 2.0 ** -51 * np.abs(psi.view(np.float64)).max() * 2.0 ** n
    diff = np.abs(got.view(np.float64) - scaled(want, e).view(np.float64))
    assert diff.max() <= np.ldexp(tol, e) + K * 2.0 ** -1021


# (Six targets take FP64 sums there, whose partial sums may overflow before the result
# does: test_gpu_six_targets.py holds them to native FP64 bit for bit.)
@pytest.mark.parametrize("n,nq,density", [(3, 20, False), (4, 18, False), (5, 18, False), (3, 5, True)])
def test_large_results(n, nq, density):
    rng = np.random.default_rng(190 + 10 * n + nq)
    size = 1 << (2 * nq if density else nq)
    psi = rng.standard_normal(size) + 1j * rng.standard_normal(size)
    mat = wl.haar_unitary(1 << n, rng)
    targs = [int(t) for t in rng.permutation(nq)[:n]]
    want = orc.run_ops(psi, [{"op": "unitary", "ctrls": [], "targs": targs, "mat": mat}], is_density=density)
    passes = 2 if density else 1
    got = apply(nq, density, targs, scaled(mat, 524 // passes), scaled(psi, 500)).view(np.float64)
    w = want.view(np.float64)
    # 2^1024 and above overflow: w from 1 on (away from the line by the error)
    big = np.abs(w) > 1.0 + 1e-12
    assert np.array_equal(got[big], np.where(w[big] > 0, np.inf, -np.inf))
    ok = np.abs(w) < 1.0 - 1e-12
    assert np.all(np.isfinite(got[ok]))
    assert np.abs(np.ldexp(got[ok], -1024) - w[ok]).max() <= 1e-13
