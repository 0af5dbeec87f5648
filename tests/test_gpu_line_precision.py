"""GPU: roundings that the line solves and what surrounds them promise."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
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


# 16 | 17 chunks a line: the last lengths whose lines store the carried pressure in the next stage's layout and the first
# ones that do not; and lengths whose lines just fit a CTA's shared memory together
@pytest.mark.parametrize("method,n,fp64", [(m, n, f) for m, n in ((CFD, 157), (CFD, 158), (MFD, 160), (MFD, 161)) for f in (True, False)]
                         + [(CFD, 122, False), (CFD, 930, True), (MFD, 150, False), (MFD, 706, False)])
def test_lines_at_layout_limits(adi, method, n, fp64):
    """The path's own tolerances: FP64 max |difference| <= 1e-12 x max |field|, FP32 relative L2 <= 1e-4."""
    rng = np.random.default_rng(n)
    for nx, ny in ((n, 24), (24, n)):
        c, *F = [rng.uniform(0.6, 1.4, wl.shapes(method, nx, ny)[0])] + [rng.standard_normal(s) for s in wl.shapes(method, nx, ny)]
        h = 1.0 / n
        dt = 0.8 * h / c.max()
        sim = adi.Sim(method, nx, ny, h, dt, c, *F, precision=adi.ADI_FP64 if fp64 else adi.ADI_FP32)
        sim.step(3)
        got = sim.read()
        sim.close()
        for g, o in zip(got, oracle.run(method, nx, ny, h, dt, c ** 2, *F, 3)):
            if fp64:
                assert np.max(np.abs(g - o)) <= 1e-12 * np.max(np.abs(o))
            else:
                assert np.linalg.norm(g - o) <= 1e-4 * np.linalg.norm(o)
