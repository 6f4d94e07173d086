"""The fixed-point form of the FP64 transforms (csrc/fx.cuh) on the CPU: the
kernels' own passes against long double sums, next to an FP64 transform of the
same input.  Bound: the error of the FP64 transform, or the rounding of the
results (2^-53) where that is larger."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2001_06113_gb300", "csrc")


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("fx") / "fx_host")
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-o", exe, os.path.join(HERE, "fx_host.cu")], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    return r.stdout.splitlines()


def test_conversions_and_products_over_their_range(lines):
    assert lines[0] == "bad 0"


def test_transform_error_is_below_the_fp64_passes(lines):
    rows = [line.split() for line in lines[1:]]
    assert len(rows) == 9 * 8 and {int(r[0]) for r in rows} == {8, 16, 32, 64, 128, 256, 512, 1024, 4096}
    for n, inv, kind, scale, fx, fp in rows:
        assert float(fx) <= max(float(fp), 2.0 ** -53), (n, inv, kind, scale, fx, fp)
