"""CPU checks of how the factored solver's records are built (no GPU needed), from the CUDA sources run on the host:
tests/reach_check.cu, the windowed scans' reach against the same products in FP64; tests/records_check.cu, the records of
lines built by several runs against extended precision; tests/lines_per_cta_check.cu, the lines that fit a CTA."""
import os
import shutil
import subprocess

import pytest

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
                        "-o", exe, os.path.join(HERE, name + ".cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "bad 0" in r.stdout, r.stdout[-2000:]


def test_reach_host_check():
    _build_and_run("reach_check")


def test_records_host_check():
    _build_and_run("records_check")


def test_lines_per_cta_host_check():
    _build_and_run("lines_per_cta_check")
