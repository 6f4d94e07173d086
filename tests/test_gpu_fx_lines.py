"""Interleaved FP64 lines of one CTA (csrc/cplx.cuh): each line has the precision of
an FP64 transform of its own, whatever the scale of its neighbours."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_lines_of_different_scales(tmp_path):
    """Bound: three roundings of the results (2^-53 / sqrt 3 each), as for single lines."""
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "lines")
    subprocess.run([nvcc, "-std=c++17", "-O3", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_2001_06113_gb300", "csrc"), "-o", exe, os.path.join(HERE, "lines_device.cu")],
                   check=True, capture_output=True)
    rows = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(rows) == 8
    for row in rows:
        assert float(row.split()[3]) <= 3.0 ** 0.5 * 2.0 ** -53, row
