"""Host check of the output scaling of the complex128 dense kernels
(paper_2311_01512_gb300/csrc/qs_bytes.cuh, driven by tests/host/scale_check.cpp).
Compiled with g++; CPU only."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_output_scaling(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path / "scale_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2311_01512_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "scale_check.cpp"), "-o", out], check=True)
    res = subprocess.run([out], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout
