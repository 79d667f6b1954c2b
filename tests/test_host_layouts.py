"""The coarse fold's shared-memory layout, the staged chunk's halving and the flat trial lists,
compiled from the library's headers and run on the CPU (tests/host_layouts.cu)."""
import os
import subprocess

import pytest

from test_host_logic import OUT_DIR, ROOT, _nvcc


def test_layouts_and_lists():
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    os.makedirs(OUT_DIR, exist_ok=True)
    exe = os.path.join(OUT_DIR, "host_layouts")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                        os.path.join(ROOT, "tests", "host_layouts.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
