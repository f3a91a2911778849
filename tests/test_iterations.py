"""Iteration counters at the end of the longest runs (I_max up to 2^32 - 1)."""
import os
import shutil
import subprocess

import pytest


def test_iteration_arithmetic(tmp_path):
    """A host-only C++ check of the functions the kernels take their loop
    bounds, schedule entries and ring fills from.  (Such runs take minutes to
    hours on a device, and an entry past the schedule's end would be a read out
    of bounds there.)"""
    gxx = shutil.which("g++")
    cuda_inc = "/usr/local/cuda/include"
    if gxx is None or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    here = os.path.dirname(os.path.abspath(__file__))
    csrc = os.path.join(os.path.dirname(here), "paper_2205_13399_gb300", "csrc")
    exe = str(tmp_path / "iteration_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", csrc, "-I", cuda_inc,
                    os.path.join(here, "iteration_check.cc"), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout
