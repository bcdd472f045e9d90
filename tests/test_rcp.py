"""The reciprocal of the PCG's scalars, built for the host: within 0.51 units of
the last place wherever it replaces the division (its step leaves 2^-68, so only
the last rounding counts), and the division's own bits elsewhere."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reciprocal_is_within_its_bound(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "rcp"
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2409_12190_gb300", "csrc"), os.path.join(ROOT, "tests", "c", "rcp.cpp"),
                    "-o", str(exe)], check=True)
    worst, differ = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert 0.49 < float(worst) <= 0.51 and int(differ) == 0
