"""Change of frame of the mixed steps' history (csrc/tables.cu) against long double
arithmetic."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_history_is_rounded_once_from_fp64_products(tmp_path):
    """Half an FP32 ulp and, for the phases, four FP64 roundings of a product."""
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    csrc = os.path.join(ROOT, "paper_2001_06113_gb300", "csrc")
    exe = str(tmp_path / "interaction")
    subprocess.run([nvcc, "-std=c++17", "-O3", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", csrc, "-I", os.path.join(ROOT, "include"), "-o", exe, os.path.join(HERE, "interaction_device.cu"),
                    os.path.join(csrc, "tables.cu")], check=True, capture_output=True)
    two, three = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert float(two) <= 2.0 ** -50 and float(three) <= 2.0 ** -50
