"""Fixed-point FP64 transforms (csrc/fx.cuh) of inputs that sit in few places of
the line, up to the longest lines, on the CPU: the kernels' passes against long
double sums.  Bound: the error of an FP64 transform of the same input, or three
roundings of the results (2^-53 / sqrt 3 each, relative to their size) where that
is larger."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2001_06113_gb300", "csrc")


def test_narrow_inputs_keep_fp64_precision(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    exe = str(tmp_path / "fx_host_long")
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-o", exe, os.path.join(HERE, "fx_host_long.cu")], check=True, capture_output=True)
    rows = [r.split() for r in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 3 * 16 + 3 * 8
    for n, inv, plan, kind, fx, fp in rows:
        assert float(fx) <= max(float(fp), 3.0 ** 0.5 * 2.0 ** -53), (n, inv, plan, kind, fx, fp)
