"""Kernel attributes are set once per device (csrc/device_once.h), on the CPU with a
fake of cudaGetDevice."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2001_06113_gb300", "csrc")


def test_set_up_runs_once_per_device(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no compiler or CUDA headers")
    exe = str(tmp_path / "device_once")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", include, "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "device_once.cpp")], check=True, capture_output=True)
    assert subprocess.run([exe], capture_output=True, text=True).stdout.strip() == "0"
