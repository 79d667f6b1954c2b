"""The handle's workspace policy on the CPU (tests/host_workspace.cu): a job that fits in its
plain form is taken whatever the buffers held before, and repeated calls allocate nothing."""
import os
import subprocess

import pytest

from test_host_logic import OUT_DIR, ROOT, _nvcc


def test_workspace_policy():
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    os.makedirs(OUT_DIR, exist_ok=True)
    exe = os.path.join(OUT_DIR, "host_workspace")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", os.path.join(ROOT, "tests", "host_workspace.cu"), "-o", exe],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
