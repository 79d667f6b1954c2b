"""The static entry's cache of launch shapes: a fixed array, so that nothing is allocated and no
exception can leave the entry point."""
import os
import re
import shutil
import subprocess

import pytest

from test_host_logic import OUT_DIR, ROOT


def test_cache():
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    os.makedirs(OUT_DIR, exist_ok=True)
    exe = os.path.join(OUT_DIR, "host_occ_cache")
    r = subprocess.run([cxx, "-O1", "-std=c++17", os.path.join(ROOT, "tests", "host_occ_cache.cc"), "-o", exe],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.returncode, r.stdout)


def test_static_entry_has_no_allocating_container():
    with open(os.path.join(ROOT, "paper_2006_06866_gb300", "csrc", "gce_static.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    assert not re.search(r"std::(map|vector|string|unordered_map|deque|list|set)\b|\bnew\b", text)
