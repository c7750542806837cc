"""Six-target complex128 gates whose matrix keeps amplitudes of a group apart
(permutations, diagonals, gates with controls of their own, entries at rounding level):
every amplitude keeps the bits that FP64 keeps, however small it is beside the others
of its group.  The bound is per output: the rounding of a sum of K products,
K 2^-53 sum_l |m_jl| |x_l| (a permutation is exact), in every way that such a pass is
made."""

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def matrix(kind, rng):
    if kind == "identity":
        return np.eye(64, dtype=np.complex128)
    if kind == "permutation":
        return np.eye(64, dtype=np.complex128)[rng.permutation(64)]
    if kind == "diagonal":
        return np.diag(np.exp(1j * rng.uniform(0, 6, 64)))
    m = np.eye(64, dtype=np.complex128)
    if kind == "controlled":
        m[32:, 32:] = wl.haar_unitary(32, rng)
    if kind == "noise":                         # zeros of a composed block at rounding level
        m[:32, :32] = wl.haar_unitary(32, rng)
        m += 1e-17 * (rng.standard_normal((64, 64)) + 1j * rng.standard_normal((64, 64)))
    return m


def spread_state(size, rng):
    v = (rng.standard_normal(size) + 1j * rng.standard_normal(size)) * 2.0 ** -rng.integers(0, 70, size=size)
    v[rng.integers(0, size, size=size // 8)] = 0.0
    return v


def check(got, psi, ops, density, unit):
    """Each pass of ops within 2 K units of sum |m| |x|, per output."""
    want = orc.run_ops(psi, ops, is_density=density)
    mags = [dict(op, mat=np.abs(op["mat"]).astype(np.complex128)) for op in ops]
    size = orc.run_ops(np.abs(psi).astype(np.complex128), mags, is_density=density).real
    passes = len(ops) * (2 if density else 1)
    assert np.all(np.abs(got - want) <= passes * 2 * 128 * unit * size)


@pytest.mark.parametrize("kind", ["identity", "permutation", "diagonal", "controlled", "noise"])
@pytest.mark.parametrize("nq,density", [(6, False), (7, False), (9, False), (14, False), (20, False), (6, True), (7, True)])
def test_passes(kind, nq, density):
    import torch
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(660 + nq)
    psi = spread_state(1 << (2 * nq if density else nq), rng)
    mat = np.ascontiguousarray(matrix(kind, rng))
    exact = kind in ("identity", "permutation")
    for ctrls in ([], [0]) if nq > 6 else ([],):
        targs = [int(t) for t in rng.permutation(nq) if t not in ctrls][:6]
        op = {"op": "unitary", "ctrls": ctrls, "targs": targs, "mat": mat}
        st = qs.State(nq, density=density, stream=torch.cuda.Stream())
        for way in ("call", "block", "program"):
            if way == "block" and ctrls:
                continue
            st.set_amps(psi)
            if way == "call":
                qs.apply_op(st.handle, op)
            elif way == "block":
                qs.qs_apply_dense_block(st.handle, targs, mat)
            else:
                qs.qs_record_begin(st.handle)
                qs.apply_op(st.handle, op)
                prog = qs.qs_record_end(st.handle)
                qs.qs_program_run(prog)
            qs.qs_synchronize(st.handle)
            got = st.get_amps()
            if way == "program":
                qs.qs_program_destroy(prog)
            if exact:
                assert np.array_equal(got, orc.run_ops(psi, [op], is_density=density)), way
            check(got, psi, [op], density, 2.0 ** -53)
        st.close()


@pytest.mark.parametrize("kind", ["permutation", "controlled"])
def test_double_float(kind):
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(67)
    psi = spread_state(1 << 13, rng)
    op = {"op": "unitary", "ctrls": [], "targs": [int(t) for t in rng.permutation(13)[:6]],
          "mat": np.ascontiguousarray(matrix(kind, rng))}
    st = qs.State(13)
    qs.qs_set_arithmetic(st.handle, qs.QS_ARITH_DF)
    st.set_amps(psi)
    qs.apply_op(st.handle, op)
    qs.qs_synchronize(st.handle)
    got = st.get_amps()
    st.close()
    check(got, psi, [op], False, 2.0 ** -46)


def test_composed_block_and_channel():
    """A fused block of NOTs with controls, and a three-qubit Kraus map of one
    permutation: both keep every bit."""
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(68)
    x = np.array([[0, 1], [1, 0]], dtype=np.complex128)
    ops = []
    for _ in range(12):
        q = [int(t) for t in rng.permutation(6)]
        ops.append({"op": "unitary", "ctrls": q[1:1 + int(rng.integers(0, 3))], "targs": q[:1], "mat": x})
    psi = spread_state(1 << 12, rng)
    st = qs.State(12)
    st.set_amps(psi)
    circ = qs.Circuit(12, ops)
    circ.plan(qs.QS_PLAN_GREEDY, 6)
    circ.apply(st.handle)
    qs.qs_synchronize(st.handle)
    assert np.array_equal(st.get_amps(), orc.run_ops(psi, ops, is_density=False))
    circ.close()
    st.close()
    rho = spread_state(1 << 10, rng)
    kraus = [np.eye(8, dtype=np.complex128)[rng.permutation(8)]]
    dm = qs.State(5, density=True)
    dm.set_amps(rho)
    qs.qs_apply_kraus(dm.handle, [3, 0, 2], kraus)
    got = dm.get_amps()
    dm.close()
    assert np.array_equal(got, orc.run_ops(rho, [{"op": "kraus", "targs": [3, 0, 2], "kraus": kraus}], is_density=True))


def gate(arith, nq, targs, ctrls, mat, psi, density=False):
    from paper_2311_01512_gb300 import qs
    st = qs.State(nq, density=density)
    qs.qs_set_arithmetic(st.handle, arith)
    st.set_amps(psi)
    qs.qs_apply_ctrl_multi_target(st.handle, ctrls, targs, mat)
    qs.qs_synchronize(st.handle)
    got = st.get_amps()
    st.close()
    return got


@pytest.mark.parametrize("nq", [6, 7, 12, 13, 14, 20])
def test_groups_out_of_range(nq):
    """With a matrix that mixes: groups that hold an infinity or a NaN, are far too
    small, or have such results come out as in native FP64, bit for bit, the others as
    without them."""
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(670 + nq)
    mat = np.ascontiguousarray(wl.haar_unitary(64, rng))
    perm = [int(t) for t in rng.permutation(nq)]
    targs = perm[:6]
    ctrls = perm[6:7] if nq > 7 else []
    size = 1 << nq
    psi = rng.standard_normal(size) + 1j * rng.standard_normal(size)
    idx = np.arange(size)
    group = idx.copy()
    for t in targs:
        group &= ~(1 << t)
    groups = np.unique(group[[(i & sum(1 << c for c in ctrls)) == sum(1 << c for c in ctrls) for i in idx]])
    values = [complex(np.inf, 1.0), complex(0.0, -np.inf), complex(np.nan, 0.0), "tiny", "large", "zero", "subnormal"]
    odd = rng.permutation(groups)[:min(len(groups), 64)]
    changed = psi.copy()
    for k, g in enumerate(odd):
        v = values[k % len(values)]
        members = idx[group == g]
        if isinstance(v, complex):
            changed[rng.choice(members)] = v
        else:
            changed[members] *= {"tiny": 2.0 ** -1000, "large": 2.0 ** 1018, "zero": 0.0, "subnormal": 2.0 ** -1030}[v]
    got = gate(qs.QS_ARITH_FX, nq, targs, ctrls, mat, changed)
    plain = gate(qs.QS_ARITH_FX, nq, targs, ctrls, mat, psi)
    native = gate(qs.QS_ARITH_F64, nq, targs, ctrls, mat, changed)
    rest = ~np.isin(group, odd)
    assert np.array_equal(got[rest].view(np.uint64), plain[rest].view(np.uint64))
    for k, g in enumerate(odd):
        if values[k % len(values)] != "large":
            m = group == g
            assert np.array_equal(got[m].view(np.float64), native[m].view(np.float64), equal_nan=True), values[k % len(values)]
    large = np.isin(group, odd[4::len(values)])
    g, w = got[large].view(np.float64), native[large].view(np.float64)
    assert np.array_equal(np.isfinite(g), np.isfinite(w))
    assert np.all(np.abs(g - w)[np.isfinite(w)] <= 1e-13 * np.float64(2.0) ** 1021)


@pytest.mark.parametrize("value", [np.inf, np.nan, complex(0, np.inf)])
def test_matrix_not_finite(value):
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(69)
    mat = np.ascontiguousarray(wl.haar_unitary(64, rng))
    mat[5, 9] = value
    psi = rng.standard_normal(1 << 9) + 1j * rng.standard_normal(1 << 9)
    args = (9, [4, 0, 7, 2, 8, 5], [], mat, psi)
    got, want = gate(qs.QS_ARITH_FX, *args), gate(qs.QS_ARITH_F64, *args)
    assert np.array_equal(got.view(np.float64), want.view(np.float64), equal_nan=True)


def test_recorded_gates_share_their_scratch():
    """Sixty recorded six-target gates need the memory of their matrices (3.8 MB, two
    chunks of the program's 4 MB with its scratch), not a scratch each (18 MB more)."""
    import torch
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(70)
    nq = 8
    psi = wl.random_statevector(nq, rng)
    ops = [{"op": "unitary", "ctrls": [], "targs": [int(t) for t in rng.permutation(nq)[:6]],
            "mat": wl.haar_unitary(64, rng) if k % 3 else matrix("controlled", rng)} for k in range(60)]
    st = qs.State(nq, stream=torch.cuda.Stream())
    st.set_amps(psi)
    qs.qs_record_begin(st.handle)
    try:
        qs.qs_test_fail_allocations(1, 100)
        for op in ops:
            qs.apply_op(st.handle, op)
    finally:
        qs.qs_test_fail_allocations(0, 0)
    prog = qs.qs_record_end(st.handle)
    want = psi
    for _ in range(2):
        qs.qs_program_run(prog)
        want = orc.run_ops(want, ops, is_density=False)
    qs.qs_synchronize(st.handle)
    assert np.max(np.abs(st.get_amps() - want)) < 1e-13
    qs.qs_program_destroy(prog)
    st.close()
