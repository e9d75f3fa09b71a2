"""The host side of the library (csrc/api.cu) on a CUDA runtime whose streams
run their work only when something ordered after it is waited for
(host_runtime.cpp): what a call must wait for, or plan, shows on the CPU."""
import os
import shutil
import subprocess

import pytest

from paper_2103_12194_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def binary(tmp_path_factory):
    nvcc = shutil.which(build.nvcc())
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc or "")), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    exe = str(tmp_path_factory.mktemp("host") / "host_runtime")
    subprocess.check_call(
        ["g++", "-std=c++17", "-O1", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
         "-I", cuda, "-x", "c++", os.path.join(build.CSRC, "api.cu"),
         os.path.join(HERE, "host_runtime.cpp"), "-o", exe])
    return exe


@pytest.mark.parametrize("scenario", ["replay_after_changes", "stream_changed_after_steps",
                                      "replays_on_the_null_stream", "device_arrays", "failed_read",
                                      "copies_on_the_null_stream"])
def test_host_side(binary, scenario):
    p = subprocess.run([binary, scenario], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout + p.stderr
