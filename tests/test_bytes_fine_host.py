"""Host check of how precisely the byte slices give back a result of at most 64 terms
(paper_2311_01512_gb300/csrc/qs_bytes.cuh, driven by tests/host/bytes_fine_check.cpp):
rows with one entry keep every bit of amplitudes near the row's largest, nothing is
one-sided, and neither they nor dense rows are further off than eight 7-bit digits
were (2.6e-17 of the row's largest amplitude, 7.0e-17 of the results' rms).  CPU only."""

import math
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_precision(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path / "bytes_fine_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2311_01512_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "bytes_fine_check.cpp"), "-o", out], check=True)
    res = subprocess.run([out], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout
    for line in res.stdout.splitlines():
        _, one, mean, dense = (float(w) for w in line.split())
        assert one <= 2.6e-17 and dense <= 7.0e-17
        assert abs(mean) <= 6 * one / math.sqrt(60000)
