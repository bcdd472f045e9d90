"""A launch refused during a stream capture fails the capture (on fakes of the
CUDA calls, no GPU): otherwise the captured trial would be replayed without it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_12190_gb300", "csrc")
TOO_LARGE, INVALIDATED = 720, 901  # cudaErrorCooperativeLaunchTooLarge, cudaErrorStreamCaptureInvalidated


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("g++ or the CUDA headers not available")
    out = tmp_path_factory.mktemp("capture") / "capture_end"
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-isystem", include, "-I", CSRC,
                    os.path.join(ROOT, "tests", "c", "capture_end.cpp"), "-o", str(out)], check=True)
    return str(out)


@pytest.mark.parametrize("refused,ended,want", [
    (0, 0, (0, 1, 0, 0)),
    (TOO_LARGE, 0, (TOO_LARGE, 0, 1, 0)),  # the graph without the refused launch is not kept
    (0, INVALIDATED, (INVALIDATED, 0, 0, 0)),
    (TOO_LARGE, INVALIDATED, (TOO_LARGE, 0, 0, 0)),
])
def test_a_refused_launch_fails_the_capture(exe, refused, ended, want):
    out = subprocess.run([exe, str(refused), str(ended)], capture_output=True, text=True, check=True).stdout
    assert tuple(int(v) for v in out.split()) == want


def test_the_trial_is_captured_with_it():
    src = open(os.path.join(CSRC, "ba_api.cu")).read()
    assert "end_capture(h->s, &g)" in src and "cudaStreamEndCapture" not in src
