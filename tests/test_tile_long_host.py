"""Schedules of long circuits take time in proportion to their gates, also when some
qubits are not used or used by a single gate only (tests/host/tile_long_check.cpp).
Compiled with g++; CPU only."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_long_circuits(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path / "tile_long_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2311_01512_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "tile_long_check.cpp"), "-o", out], check=True)
    res = subprocess.run([out], capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stdout
    seconds = [float(line.split()[0]) for line in res.stdout.splitlines()]
    # scanning every gate left for every pass takes a hundred times as long
    assert seconds[1] < 10 * seconds[0] and seconds[2] < 10 * seconds[0], seconds
