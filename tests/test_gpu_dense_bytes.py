"""Complex128 dense gates on the byte-sliced tensor-core kernels at the edges of
their tiles: fewer groups than a tile's 128 rows, passes of fewer tiles than SMs and of
many per CTA (the rings' phases go round several times), controls, amplitudes and matrices of widely
spread magnitudes, and the conjugate and superoperator passes of density
matrices.  All outputs against the oracle within a bound on the whole state, and the
outputs of sampled groups against extended precision within the kernel's own bound on
their group."""

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


SMALL = {2: 20, 3: 19, 4: 17, 5: 17}     # passes over at most 2^SMALL amplitudes take k_dense_fx


def parts(z):
    return np.stack([z.real, z.imag], axis=-1)


def exponent(v):
    """Exponent that the byte slices scale by (qs_bytes.cuh): one more from 2 - 2^-7 on."""
    e = np.frexp(v)[1] - 1
    return np.where(np.ldexp(v, -e) >= 2 - 2.0 ** -7, e + 1, e)


def kernel_bound(n, size, x, mat, y):
    """Error bound of the parts of y = mat x, x of shape (amplitudes, groups): the bounds
    stated at the kernels, in terms of each group's largest part and each row's."""
    big = np.abs(parts(x)).max(axis=(0, 2))[None, :, None]
    row = np.abs(parts(mat)).max(axis=(1, 2))[:, None, None]
    least = np.abs(parts(mat)).max(axis=2).min(axis=1)[:, None, None]
    rounding = 2.0 ** -53 * np.abs(parts(y))
    if n == 6 and np.any(least < row * 2.0 ** -15):            # FP64 sums (2^-16 is the kernel's line)
        return 128 * 2.0 ** -53 * (np.abs(mat) @ np.abs(x))[:, :, None] + rounding
    if n < 6 and size <= SMALL[n]:
        return rounding + (2 ** (n + 4) + (2 ** (2 * n - 2) if n > 2 else 0)) * 2.0 ** -60 * big * row
    K, X = max(16, 2 << n), 0 if n == 6 else 2
    ea, eb = np.where(big > 0, exponent(big), -2000), np.where(row > 0, exponent(row), -2000)
    sums = np.abs(parts(mat)).sum(axis=(1, 2))[:, None, None]
    return (rounding + np.ldexp(sums * (0.5 + 2.0 ** -8), ea - 54) + np.ldexp(K, ea + eb - 62) +
            np.ldexp(0.6 + 6 * K * 2.0 ** (X - 10), ea + eb - 52 - X))


def groups(nq, targs, ctrls, count, rng):
    """Indices (amplitudes, groups) of randomly chosen groups of a gate."""
    free = [q for q in range(nq) if q not in targs and q not in ctrls]
    g = np.unique(rng.integers(0, 1 << len(free), size=count))
    base = sum(1 << c for c in ctrls) + sum(((g >> b) & 1) << q for b, q in enumerate(free))
    l = np.arange(1 << len(targs))
    return sum(((l >> b) & 1) << t for b, t in enumerate(targs))[:, None] + (base + 0 * g)[None, :]


def extended(mat, x):
    """Parts of mat x in extended precision."""
    m, v = parts(mat).astype(np.longdouble), parts(x).astype(np.longdouble)
    y = np.zeros(x.shape + (2,), dtype=np.longdouble)
    for l in range(mat.shape[1]):
        mr, mi, xr, xi = m[:, l, 0][:, None], m[:, l, 1][:, None], v[l, :, 0][None, :], v[l, :, 1][None, :]
        y[..., 0] += mr * xr - mi * xi
        y[..., 1] += mr * xi + mi * xr
    return y


def errors(got, psi, nq, targs, ctrls, mat, rng, count=96):
    """Errors of sampled groups, each within its bound; and the exact parts."""
    at = groups(nq, targs, ctrls, count, rng)
    x, exact = psi[at], extended(np.asarray(mat), psi[at])
    e = (parts(got[at]) - exact).astype(np.float64)
    limit = kernel_bound(len(targs), nq - len(ctrls), x, np.asarray(mat), exact[..., 0] + 1j * exact[..., 1])
    assert np.all(np.abs(e) <= limit.astype(np.float64)), np.max(np.abs(e) / np.maximum(limit, 1e-300))
    return e, exact


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
        errors(got, psi, nq, targs, ctrls, mat, rng)


@pytest.mark.parametrize("n,nq", [(2, 12), (2, 21), (3, 12), (3, 20), (4, 12), (4, 18), (5, 12), (5, 18), (6, 12)])
def test_average_error(n, nq):
    """On both sides of the size where passes change kernel: the error in the 2-norm, at
    most that of the 7-bit digits that these kernels replaced (7.7, 6.6, 7.6e-17 for 3 to 5
    targets, two ran as three; FP64 37e-17 at six) and in fact below 6.7e-17, with hardly
    a one-sided part.  (Amplitudes with one to a few bits below their unit of 2^-54 tie and
    go up: 0.06 units on average, 0.15 of one output's rms error times the sum of its row,
    whose signs differ among the 2^(n + 1) outputs; sums rounded down had 0.6 to 0.9.)"""
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(5000 + 10 * n + nq)
    psi = wl.random_statevector(nq, rng)
    mat = np.ascontiguousarray(wl.haar_unitary(1 << n, rng))
    targs = [int(t) for t in rng.permutation(nq)[:n]]
    st = qs.State(nq)
    st.set_amps(psi)
    qs.qs_apply_dense_block(st.handle, targs, mat)
    got = st.get_amps()
    st.close()
    if n == 2 and nq > SMALL[2]:                # runs as three, with an identity on the lowest free qubit
        targs, mat = targs + [min(set(range(nq)) - set(targs))], np.kron(np.eye(2), mat)
    e, exact = errors(got, psi, nq, targs, [], mat, rng, 8192 >> n)
    assert np.linalg.norm(e) <= 6.7e-17 * np.linalg.norm(exact.astype(np.float64))
    assert abs(e.mean()) <= 0.1 * e.std()


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
        if n > 2 or not ctrls:                  # (two targets with controls: k_gate2_fx)
            errors(got, psi, nq, perm[:n], ctrls, mat, rng)


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
