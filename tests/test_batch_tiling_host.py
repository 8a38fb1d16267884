"""A tile shape that fdlb_autotune returned gives the tuned grid again when it
is set with fdlb_batch_set_tiling (as a program does that saves the result).
The host code runs on a stand-in for the CUDA runtime (tests/host/tiling_host.cpp)."""
import os
import subprocess

import pytest

from test_host_sanitizers import BUILD, HERE, ROOT, _cuda_home


def test_a_tuned_shape_can_be_set_again():
    cuda = _cuda_home()
    if not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("CUDA headers not found")
    os.makedirs(BUILD, exist_ok=True)
    exe = os.path.join(BUILD, "tiling_host")
    csrc = os.path.join(ROOT, "paper_1909_08390_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-I",
                    os.path.join(cuda, "include"), os.path.join(HERE, "host", "tiling_host.cpp"),
                    os.path.join(csrc, "fdlb_api.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr
