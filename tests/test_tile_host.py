"""Host check of the tile passes of circuits (paper_2311_01512_gb300/csrc/qs_tile.h,
driven by tests/host/tile_check.cpp): the schedule and the kernel's index arithmetic
against the gates one by one.  The matrices are FP32 values and the sums FP64, so
only the gadgets' cosines and sines, rounded to FP32 (2^-25 relative each, at most
60 gates, each at most twice the amplitude's size), differ.  CPU only."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tile_passes(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path / "tile_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2311_01512_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "tile_check.cpp"), "-o", out], check=True)
    res = subprocess.run([out], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout
    assert float(res.stdout) <= 60 * 2 * 2.0 ** -25
