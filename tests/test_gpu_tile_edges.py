"""GPU: the sizes at which the step's kernels change their path or their tiles end, against the FP64 CPU oracle.

Tolerances are the path's own (FP64 max |difference| <= 1e-12 x max |field|, FP32 relative L2 <= 1e-4), for
the few steps taken here; where two GPU paths are compared they are derived beside the test.
"""
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


def _case(method, nx, ny, seed, cfl=0.8):
    rng = np.random.default_rng(seed)
    su, sv, sw = wl.shapes(method, nx, ny)
    h = 1.0 / max(nx, ny)
    c = rng.uniform(0.6, 1.4, su)
    U, V, W = rng.standard_normal(su), rng.standard_normal(sv), rng.standard_normal(sw)
    return h, cfl * h / c.max(), c, U, V, W


def _check(got, want, fp64):
    for g, o in zip(got, want):
        if fp64:
            assert np.max(np.abs(g - o)) <= 1e-12 * np.max(np.abs(o))
        else:
            assert np.linalg.norm(g - o) <= 1e-4 * np.linalg.norm(o)


# chunks per line on either side of: 32 | 33 (a line within a warp), 64 | 65 (end rows by the middle warps), 192 |
# 193 and 224 | 225 (one row per lane or per half-warp; FP64 CTAs of 256 or 512 threads), and the last line lengths
# of an MFD remainder of 0, 1 and 2 blocks; chunks are 9 nodes (CFD, N - 5 of them) or 9 cells (MFD, about N - 8)
LINES = [(CFD, 5 + 9 * 32), (CFD, 5 + 9 * 33), (CFD, 5 + 9 * 64 + 8), (CFD, 5 + 9 * 65), (CFD, 5 + 9 * 192),
         (CFD, 5 + 9 * 193), (CFD, 5 + 9 * 224 + 8), (CFD, 5 + 9 * 225), (MFD, 16), (MFD, 17), (MFD, 8 + 9 * 32),
         (MFD, 8 + 9 * 33 + 4), (MFD, 8 + 9 * 65 + 7), (MFD, 8 + 9 * 193), (MFD, 8 + 9 * 224 + 8), (MFD, 8 + 9 * 225 + 1)]


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("method,n", LINES)
def test_line_lengths_at_path_changes(adi, method, n, fp64):
    nx, ny = (n, 20) if n % 2 else (20, n)  # the long lines along x or y
    h, dt, c, U, V, W = _case(method, nx, ny, n)
    src = (ny // 2, nx // 3, 0.01, 15.0, 0.0)
    sim = adi.Sim(method, nx, ny, h, dt, c, U, V, W, precision=adi.ADI_FP64 if fp64 else adi.ADI_FP32)
    assert sim.solver == adi.ADI_SOLVER_FACTORED
    sim.set_source(*src)
    sim.step(3)
    G = sim.read()
    sim.close()
    _check(G, oracle.run(method, nx, ny, h, dt, c ** 2, U, V, W, 3, source=src), fp64)


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("method,nx,ny", [(CFD, 33, 31), (CFD, 40, 32), (CFD, 31, 33), (CFD, 65, 64), (CFD, 34, 95),
                                          (CFD, 31, 97), (CFD, 33, 130), (MFD, 33, 31), (MFD, 64, 66)])
def test_loading_fields_mid_run(adi, method, nx, ny, fp64):
    """New fields loaded into a simulation that has stepped an odd number of steps: the carried state is rebuilt
    from them (chunks of 32 rows of every line) and nothing of the old fields is left in the arrays."""
    h, dt, c, U, V, W = _case(method, nx, ny, 7)
    U2, V2, W2 = _case(method, nx, ny, 8)[3:]
    sim = adi.Sim(method, nx, ny, h, dt, c, U, V, W, precision=adi.ADI_FP64 if fp64 else adi.ADI_FP32)
    sim.step(3)
    if fp64:
        sim.set_fields(U2, V2, W2)
    else:
        sim.set_fields_f32(*[np.ascontiguousarray(a, dtype=np.float32) for a in (U2, V2, W2)])
    _check(sim.read(), (U2, V2, W2), fp64)
    sim.step(2)
    G = sim.read()
    sim.close()
    _check(G, oracle.run(method, nx, ny, h, dt, c ** 2, U2, V2, W2, 2), fp64)


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("method,nx,ny,layers", [(CFD, 40, 33, 0), (MFD, 33, 143, 0), (MFD, 144, 30, 0), (CFD, 143, 31, 4),
                                                 (CFD, 31, 300, 0)])
def test_short_lines_alone_and_in_a_wide_batch(adi, method, nx, ny, layers, fp64):
    """Lines of up to 15 chunks store the carried pressure in the next stage's layout at once when their launch is one
    round of groups, as for the simulation alone, and in their own layout beside members that make it two (CFD and
    MFD of 1030 cells, whose solves also run on two streams): the steps before, in and after such a batch."""
    h, dt, c, U, V, W = _case(method, nx, ny, 31)
    prec = adi.ADI_FP64 if fp64 else adi.ADI_FP32
    src = (ny // 2, nx // 3, 0.01, 15.0, 0.0)
    sims = [adi.Sim(method, nx, ny, h, dt, c, U, V, W, precision=prec)]
    sims[0].set_source(*src)
    if layers:
        sims[0].set_sponge(layers, 0.1)
    for m in (CFD, MFD):
        bh, bdt, bc, bU, bV, bW = _case(m, 1030, 1030, 32)
        sims.append(adi.Sim(m, 1030, 1030, bh, bdt, bc, bU, bV, bW, precision=prec))
    sims[0].step(1)
    b = adi.Batch(sims)
    b.step(3)
    b.sync()
    b.close()
    mid = sims[0].read()
    sims[0].step(2)
    end = sims[0].read()
    for s in sims:
        s.close()
    for got, n in ((mid, 4), (end, 6)):
        if layers:
            want = oracle.run_sponge(method, nx, ny, h, dt, c ** 2, U, V, W, n, layers, 0.1, source=src)
        else:
            want = oracle.run(method, nx, ny, h, dt, c ** 2, U, V, W, n, source=src)
        _check(got, want, fp64)


# line counts around a block's four lines; lines so long that a block takes two (FP64 above about 7230 cells, FP32 above
# 14460) or one (FP64 above 14460; 14522 would fit twice but for the block's other shared memory); the recurrences go
# sixteen rows at a time
@pytest.mark.parametrize("method,nx,ny,fp64", [(CFD, 16, 17, True), (CFD, 17, 18, False), (MFD, 18, 19, True),
                                               (CFD, 23, 24, True), (CFD, 25, 320, False), (CFD, 7300, 16, True),
                                               (CFD, 16, 14600, True), (MFD, 15000, 16, False),
                                               (CFD, 14522, 16, True)])
def test_fixed_point_blocks(adi, method, nx, ny, fp64):
    h, dt, c, U, V, W = _case(method, nx, ny, 21, cfl=0.6)
    src = (ny // 2, nx // 3, 0.01, 15.0, 0.0)
    *G, sweeps, _ = adi.fixed_point(method, nx, ny, h, dt, c, U, V, W, 2, source=src, kmax=3, eps=0.0,
                                    precision=adi.ADI_FP64 if fp64 else adi.ADI_FP32)
    assert sweeps == 2 * 2 * 3
    _check(G, oracle.run(method, nx, ny, h, dt, c ** 2, U, V, W, 2, source=src, kmax=3, eps=0.0), fp64)


@pytest.mark.parametrize("method", [CFD, MFD])
@pytest.mark.parametrize("cfl", [0.8, 40.0])
def test_records_of_long_lines(adi, method, cfl):
    """The factored solver's records of a line are built by several threads, each from a start that forgets what lies
    before it; with a large time step it does not and the line is done in one run.  Both against the
    thread-per-line elimination in FP64.  Tolerance: the line systems' condition number grows as cfl^2 (about 10
    at 0.8, 2e4 at 40 on these media) times a few hundred roundings of 1.1e-16: 1e-12 and 2e-9."""
    nx, ny = 2000, 40
    h, dt, c, U, V, W = _case(method, nx, ny, 5, cfl=cfl)
    out = []
    for solver in (adi.ADI_SOLVER_FACTORED, adi.ADI_SOLVER_LINE):
        sim = adi.Sim(method, nx, ny, h, dt, c, U, V, W, precision=adi.ADI_FP64, solver=solver)
        assert sim.solver == solver
        sim.step(1)
        out.append(sim.read())
        sim.close()
    tol = 1e-12 if cfl < 1 else 2e-9
    for a, b in zip(*out):
        assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b))


def test_fp64_reciprocal():
    """The FP64 line kernels' reciprocal (fac_rcp) against CUDA's correctly rounded 1 / x: at most one unit in the
    last place off, for 2^20 values over the exponents that pivots and determinants take."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = os.path.join(HERE, "_build")  # git-ignored
    os.makedirs(out, exist_ok=True)
    exe = os.path.join(out, "fac_rcp_check")
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I" + os.path.join(ROOT, "include"),
                        "-o", exe, os.path.join(HERE, "fac_rcp_check.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "worst" in r.stdout, r.stdout[-500:] + r.stderr[-500:]
    assert int(r.stdout.split()[1]) <= 1, r.stdout
