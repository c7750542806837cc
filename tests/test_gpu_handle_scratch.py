"""Memory of destroyed handles is used again by later ones: it is given back with
the last handle, bounded, carries nothing over from one handle to the next, and
may change stream and thread."""

import threading

import numpy as np
import pytest

from oracle import qsim_oracle as orc
from paper_2311_01512_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_bounded_and_given_back():
    import torch
    from paper_2311_01512_gb300 import qs
    v = torch.zeros(256, dtype=torch.complex128, device="cuda")
    qs.State(8, storage=v).close()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    states = [qs.State(8, storage=v) for _ in range(32)]
    torch.cuda.synchronize()
    many = free0 - torch.cuda.mem_get_info()[0]
    for s in states[1:]:
        s.close()
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= many / 2
    states[0].close()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free0


def test_nothing_carried_over():
    import torch
    from paper_2311_01512_gb300 import qs
    rng = np.random.default_rng(1)
    keep = qs.State(3)
    a = qs.State(4)
    qs.qs_test_set_error_word(a.handle)
    a.close()
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream()):
        b = qs.State(9, stream=stream)
        psi = wl.random_statevector(9, rng)
        b.set_amps(psi)
        qs.qs_synchronize(b.handle)                       # a's error word is not b's
        u = wl.haar_unitary(64, rng)                      # through the ring
        qs.qs_apply_ctrl_multi_target(b.handle, [], [0, 2, 3, 5, 7, 8], u)
        want = orc.apply_ctrl_multi_target(psi, [], [0, 2, 3, 5, 7, 8], u)
        assert np.max(np.abs(b.get_amps() - want)) < 1e-13
        b.close()
    keep.close()


def test_threads_and_streams():
    import torch
    from paper_2311_01512_gb300 import qs
    keep = qs.State(3)
    torch.cuda.synchronize()
    errors = []

    def work(seed):
        try:
            rng = np.random.default_rng(seed)
            for i in range(12):
                with torch.cuda.device(0):
                    st = qs.State(10, stream=torch.cuda.Stream())
                    psi = wl.random_statevector(10, rng)
                    st.set_amps(psi)
                    u = wl.haar_unitary(64, rng)
                    t = [int(q) for q in rng.permutation(10)[:6]]
                    for _ in range(3):
                        qs.qs_apply_ctrl_multi_target(st.handle, [], t, u)
                        psi = orc.apply_ctrl_multi_target(psi, [], t, u)
                    norm = qs.qs_calc_norm_or_trace(st.handle)
                    assert abs(norm - orc.calc_norm(psi)) < 1e-13
                    assert np.max(np.abs(st.get_amps() - psi)) < 1e-13
                    st.close()
        except Exception as e:                            # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    keep.close()
    assert not errors, errors
