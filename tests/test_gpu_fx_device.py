"""Device arithmetic of the FP64 and conversion paths against CUDA's own: the
reciprocal of the implicit solve (csrc/step_common.cuh) and the integer
conversions between FP32 and FP64 (csrc/fx.cuh)."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("fx") / "fx_device")
    subprocess.run([nvcc, "-std=c++17", "-O3", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_2001_06113_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-o", out, os.path.join(HERE, "fx_device.cu")], check=True, capture_output=True)
    return out


def test_reciprocal_of_the_implicit_solve(exe):
    """One step of Halley's iteration cubes the estimate's error e: with e below
    2^-18 the result is off by 2^-54 and a rounding, one ulp of 1.0 / d at most."""
    ulps, estimate, wrong = subprocess.run([exe, "recip"], capture_output=True, text=True, check=True).stdout.split()
    assert float(estimate) <= 2.0 ** -18
    assert float(ulps) <= 1.0
    assert int(wrong) == 0


def test_conversions_round_to_nearest(exe):
    """FP32 -> FP64 exact (pairs as integers and back too), FP64 -> FP32 to nearest, over
    subnormals, infinities and NaN."""
    assert subprocess.run([exe, "float"], capture_output=True, text=True, check=True).stdout.split() == ["0", "0"]
