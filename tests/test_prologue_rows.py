"""CPU: tests/prologue_rows_check.cu runs the prologue kernel's windows on the host for every line of 16 to 4096 cells, and
tests/static_prologue_check.cu measures the error of those of the allocation-free step (no GPU needed).  GPU: fields loaded into CFD grids around the first windows with constant factors."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_2006_07583_gb300 import workloads as wl

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _build_and_run(name):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = os.path.join(HERE, "_build")  # git-ignored
    os.makedirs(out, exist_ok=True)
    exe = os.path.join(out, name)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I" + os.path.join(ROOT, "include"),
                        "-diag-suppress", "20011,20013,20014", "-o", exe, os.path.join(HERE, name + ".cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "bad 0" in r.stdout, r.stdout[-2000:]


def test_prologue_rows_host_check():
    _build_and_run("prologue_rows_check")


def test_static_prologue_error_host_check():
    _build_and_run("static_prologue_check")


# P has such a window from ny = 160 on (its rows 64 to 127), Pbar from 162 on; 224 | 226 give a second one, and 208 is
# the last length whose first window ends within 16 rows of the line's end
@pytest.mark.gpu
@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("ny", [159, 160, 161, 162, 163, 208, 224, 226])
def test_loading_fields_into_long_lines(ny, fp64):
    """As after any load of fields: FP64 max |difference| <= 1e-12 x max |field|, FP32 relative L2 <= 1e-4."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_07583_gb300 import adi

    nx, rng = 33, np.random.default_rng(ny)
    h = 1.0 / ny
    c, *F = [rng.uniform(0.6, 1.4, wl.shapes(wl.CFD, nx, ny)[0])] + [rng.standard_normal(s) for s in wl.shapes(wl.CFD, nx, ny)]
    dt = 0.8 * h / c.max()
    sim = adi.Sim(wl.CFD, nx, ny, h, dt, c, precision=adi.ADI_FP64 if fp64 else adi.ADI_FP32)
    sim.step(1)
    sim.set_fields(*F)
    sim.step(2)
    got = sim.read()
    sim.close()
    for g, o in zip(got, oracle.run(wl.CFD, nx, ny, h, dt, c ** 2, *F, 2)):
        if fp64:
            assert np.max(np.abs(g - o)) <= 1e-12 * np.max(np.abs(o))
        else:
            assert np.linalg.norm(g - o) <= 1e-4 * np.linalg.norm(o)
