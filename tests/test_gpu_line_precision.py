"""GPU: roundings that the line solves and what surrounds them promise."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2006_07583_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CFD, MFD = wl.CFD, wl.MFD
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


@pytest.mark.parametrize("method,nx,ny", [(CFD, 40, 33), (MFD, 100, 140)])
def test_natural_pressure_of_subnormal_fields(adi, method, nx, ny):
    """u = (a + C) / 2 is rounded once wherever a is stored: for fields of a few hundred times the smallest FP32 value
    the same bits alone (lines that store a in the next stage's layout) and beside members that make the launch
    more than one round of groups (a in its own layout)."""
    got = []
    for beside in (False, True):
        rng = np.random.default_rng(3)
        c, *F = [rng.uniform(0.6, 1.4, wl.shapes(method, nx, ny)[0])] + [
            rng.standard_normal(s) * 300 * 2.0 ** -149 for s in wl.shapes(method, nx, ny)]
        sims = [adi.Sim(method, nx, ny, 1.0 / 40, 0.5 / 40, c, *F, precision=adi.ADI_FP32)]
        if beside:
            big = np.ones(wl.shapes(method, 1030, 1030)[0])
            sims.append(adi.Sim(method, 1030, 1030, 1.0 / 1030, 0.5 / 1030, big, precision=adi.ADI_FP32))
        b = adi.Batch(sims)
        b.step(2)
        b.sync()
        b.close()
        got.append([a.astype(np.float32) for a in sims[0].read()])
        for s in sims:
            s.close()
    for alone, shared in zip(*got):
        assert np.count_nonzero(alone) > alone.size // 2
        assert np.array_equal(alone.view(np.uint32), shared.view(np.uint32))
