"""GPU: roundings that the line solves and what surrounds them promise."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def adi():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_07583_gb300 import adi as _adi

    _adi.lib()
    return _adi


def test_fp64_block_inverse_divides(adi):
    """CFD's FP64 blocks are inverted with a correctly rounded division: the same bits (tests/fac_inv_check.cu)."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = os.path.join(HERE, "_build")  # git-ignored
    os.makedirs(out, exist_ok=True)
    exe = os.path.join(out, "fac_inv_check")
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I" + os.path.join(ROOT, "include"),
                        "-o", exe, os.path.join(HERE, "fac_inv_check.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "differ 0\n", r.stdout[-500:] + r.stderr[-500:]
