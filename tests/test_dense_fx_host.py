"""Host check of the dense gates of small statevectors in block fixed point
(k_dense_fx; its sums are those of paper_2311_01512_gb300/csrc/qs_fx.cuh) against
exact rational arithmetic, 2 to 5 targets, rows of Haar unitaries.

* every output within the kernel's bound;
* no one-sided error: the mean signed error of n outputs is within six standard
  errors of zero (the spread of one output is at most 1e-16 of the outputs' rms);
* on average no further off than the tensor-core kernels that take the same gate on
  larger states (6.6e-17 of the outputs' rms).
CPU only."""

import math
import os
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2311_01512_gb300 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("dense_fx") / "dense_fx_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2311_01512_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "dense_fx_check.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("spread", [0, 12])
@pytest.mark.parametrize("n", [2, 3, 4, 5])
def test_rows(exe, n, spread):
    rng = np.random.default_rng(5300 + 10 * n + spread)
    d, rows = 1 << n, []
    while len(rows) < 3000:
        x = (rng.standard_normal(d) + 1j * rng.standard_normal(d)) * 2.0 ** -rng.integers(0, spread + 1, size=d)
        for row in wl.haar_unitary(d, rng)[:4]:
            rows.append((x.view(np.float64), np.ascontiguousarray(row).view(np.float64)))
    text = "\n".join(" ".join([str(n)] + ["%016x" % bits(float(v)) for v in np.concatenate(r)]) for r in rows)
    res = subprocess.run([exe], input=text + "\n", capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr
    got = [struct.unpack("<d", struct.pack("<Q", int(w, 16)))[0] for w in res.stdout.split()]
    assert len(got) == len(rows)
    err, exact = [], []
    for (x, m), y in zip(rows, got):
        sign = (1, -1) * d
        want = sum(s * Fraction(a) * Fraction(b) for s, a, b in zip(sign, x.tolist(), m.tolist()))
        e = Fraction(y) - want
        units = 2 ** (n + 4) + (2 ** (2 * n - 2) if n > 2 else 0)
        bound = Fraction(1, 2 ** 53) * abs(want) + units * Fraction(np.abs(x).max()) * Fraction(np.abs(m).max()) / 2 ** 60
        assert abs(e) <= bound, (n, float(e), float(bound))
        err.append(float(e))
        exact.append(float(want))
    rms = math.sqrt(sum(v * v for v in exact) / len(exact))
    assert abs(sum(err)) / len(err) <= 6 * 1e-16 / math.sqrt(len(err)) * rms
    assert math.sqrt(sum(e * e for e in err) / len(err)) <= 6.6e-17 * rms
