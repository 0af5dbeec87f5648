"""CPU: the library's host code on a CUDA runtime without a GPU (tests/fake_cudart.cpp), where allocations fail, waits run
out and copies stay queued until their stream is waited for."""
import ctypes as ct
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2006_07583_gb300 import build as _build

HERE = os.path.dirname(os.path.abspath(__file__))
CFD, MFD, FP32, FP64 = 0, 1, 0, 1
OK, EINVAL, ENOMEM, ECUDA, ETIMEOUT = 0, 1, 2, 3, 5


@pytest.fixture(scope="module")
def lib():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    _build.build()
    out = os.path.join(HERE, "_build")  # git-ignored
    os.makedirs(out, exist_ok=True)
    so = os.path.join(out, "libadi_host.so")
    objs = [os.path.join(_build.BUILD, os.path.basename(s)[:-3] + ".o") for s in _build.sources()]
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + inc, "-Wl,-Bsymbolic", "-o", so,
                        os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    lib = ct.CDLL(so)
    lib.fake_last_smem.restype = ct.c_longlong
    return lib


def _ptr(a):
    return a.ctypes.data_as(ct.c_void_p)


def _sim(lib, method, nx, ny, precision):
    n = (nx + 1) * (ny + 1) if method == CFD else (nx + 2) * (ny + 2)
    c, h = np.ones(n), ct.c_void_p()
    assert lib.adi_create(ct.byref(h), method, nx, ny, ct.c_double(1.0 / nx), ct.c_double(0.5 / nx), _ptr(c), None, None,
                          None, precision) == OK
    return h


def _arrays(method, nx, ny, dtype):
    if method == CFD:
        shapes = [(ny + 1, nx + 1)] * 3
    else:
        shapes = [(ny + 2, nx + 2), (ny + 2, nx + 1), (ny + 1, nx + 2)]
    return [np.full(s, 7.0, dtype) for s in shapes]


@pytest.mark.parametrize("method", [CFD, MFD])
@pytest.mark.parametrize("precision", [FP32, FP64])
@pytest.mark.parametrize("f32", [False, True])
def test_read_without_staging_memory_leaves_nothing_behind(lib, method, precision, f32):
    """The staging buffer's allocation fails: no copy into the caller's arrays is on its way when the call returns, and
    none was made.  The handle stays usable."""
    h = _sim(lib, method, 20, 18, precision)
    read = lib.adi_read_fields_f32 if f32 else lib.adi_read_fields
    out = _arrays(method, 20, 18, np.float32 if f32 else np.float64)
    lib.fake_fail_alloc(0)
    rc = read(h, *[_ptr(a) for a in out])
    lib.fake_fail_alloc(-1)
    assert rc == ENOMEM
    assert lib.fake_host_writes() == 0
    lib.fake_run_all()
    assert all((a == 7.0).all() for a in out)
    assert read(h, *[_ptr(a) for a in out]) == OK
    assert all((a == 0.0).all() for a in out)
    assert lib.adi_destroy(h) == OK


@pytest.mark.parametrize("launch", [0, 1, 2])
def test_read_error_leaves_no_copy_on_its_way(lib, launch):
    """A conversion's launch fails after other fields' copies were queued: they have ended when the call returns."""
    h = _sim(lib, MFD, 20, 18, FP32)
    out = _arrays(MFD, 20, 18, np.float64)
    lib.fake_fail_launch(launch)
    rc = lib.adi_read_fields(h, *[_ptr(a) for a in out])
    lib.fake_fail_launch(-1)
    assert rc == ECUDA
    assert lib.fake_host_writes() == 0
    assert lib.adi_destroy(h) == OK


@pytest.mark.parametrize("method", [CFD, MFD])
@pytest.mark.parametrize("precision", [FP32, FP64])
@pytest.mark.parametrize("f32", [False, True])
def test_read_after_a_timeout_leaves_the_arrays_alone(lib, method, precision, f32):
    """A solve's bounded wait ran out: the read says so and the caller's arrays hold what they held, in the first call
    and in later ones; a simulation whose solves ended reads as usual."""
    read = lib.adi_read_fields_f32 if f32 else lib.adi_read_fields
    for fault in (0, 1):
        h = _sim(lib, method, 20, 18, precision)
        out = _arrays(method, 20, 18, np.float32 if f32 else np.float64)
        lib.fake_raise_fault(fault)
        assert lib.adi_step(h, 1) == OK
        lib.fake_raise_fault(0)
        for _ in range(2):
            assert read(h, *[_ptr(a) for a in out]) == (ETIMEOUT if fault else OK)
            lib.fake_run_all()
            assert all((a == (7.0 if fault else 0.0)).all() for a in out)
        assert lib.adi_destroy(h) == OK


@pytest.mark.parametrize("precision", [FP32, FP64])
@pytest.mark.parametrize("method", [CFD, MFD])
def test_fixed_point_keeps_its_shared_memory_limit(lib, method, precision):
    """The dynamic shared memory limit of a kernel belongs to the process: a call with short lines leaves it where a
    call with long lines, which another thread may be in the middle of, needs it."""
    for n in (4000, 16):
        shapes = [a.shape for a in _arrays(method, n, 16, np.float64)]
        c, u, v, w = [np.ones(s) for s in shapes[:1] + shapes]
        sweeps, ms = ct.c_longlong(), ct.c_double()
        rc = lib.adi_fixed_point(method, n, 16, ct.c_double(1.0 / n), ct.c_double(0.1 / n), _ptr(c), _ptr(u), _ptr(v), _ptr(w), 1,
                                 ct.c_double(0.0), None, 2, ct.c_double(0.0), precision, ct.byref(sweeps), ct.byref(ms))
        assert rc == OK
        for kernel in (b"fp_sweep_kernel", b"fp_rhs_kernel"):
            name = kernel + (b"IdE" if precision == FP64 else b"IfE")
            limit, used = ct.c_longlong(), ct.c_longlong()
            lib.fake_smem(name, ct.byref(limit), ct.byref(used))
            assert limit.value >= used.value >= 48 * 1024


@pytest.mark.parametrize("precision,kernel", [(FP32, b"IfLi2ELi9ELb0E"), (FP64, b"IdLi2ELi9ELb0E")])
def test_line_solves_keep_their_shared_memory_limit(lib, precision, kernel):
    """The same for the factored solver's launches: simulations of different sizes are stepped from several threads."""
    for n in (4000, 16):
        h = _sim(lib, CFD, n, 16, precision)
        assert lib.adi_step(h, 1) == OK and lib.adi_sync(h) == OK and lib.adi_destroy(h) == OK
        limit, used = ct.c_longlong(), ct.c_longlong()
        lib.fake_smem(b"line_solve_factored_kernel" + kernel, ct.byref(limit), ct.byref(used))
        assert limit.value >= used.value >= 48 * 1024


def test_autotune_leaves_the_chosen_launch(lib):
    """Every candidate takes the same time here, so the automatic launch is chosen; the steps after the call run it and
    not the last one tried, the first time and from the cached choice."""
    def smem_of_a_step(h):
        assert lib.adi_step(h, 1) == OK and lib.adi_sync(h) == OK
        return lib.fake_last_smem(b"line_solve_factored_kernelIfLi2ELi9ELb0E")

    sims = [_sim(lib, CFD, 100, 100, FP32) for _ in range(3)]
    want = smem_of_a_step(sims[0])
    for h in sims[1:]:
        chosen, cap, ring = ct.c_int(-1), ct.c_int(-1), ct.c_int(-1)
        assert lib.adi_autotune(h, 2, 0, ct.byref(chosen), None) == OK
        assert lib.adi_get_launch(h, ct.byref(cap), ct.byref(ring)) == OK
        assert (chosen.value, cap.value, ring.value) == (2, 0, 0)
        assert smem_of_a_step(h) == want
    for h in sims:
        assert lib.adi_destroy(h) == OK
