"""Fixed-point conversions (csrc/fx.cuh) at the lower end of the FP64 range, on the
CPU: nothing that FP64 holds is dropped, subnormals among it."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2001_06113_gb300", "csrc")


def test_small_values_are_kept(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    exe = str(tmp_path / "fx_host_range")
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-o", exe, os.path.join(HERE, "fx_host_range.cu")], check=True, capture_output=True)
    first, *rows = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines()
    assert first == "0 0 0"
    # the same integers come out of the passes; their rounding to FP64 differs by one step at most
    assert len(rows) == 6
    for row in rows:
        assert float(row.split()[1]) <= 1.0, row
