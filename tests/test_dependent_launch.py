"""Kernels that are launched while the one before them still runs promise nothing about memory
that it writes: `const __restrict__` (which lets loads go through the non-coherent path and
ahead of the wait) is for the caller's arrays alone."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CALLERS = {"times", "mags", "periods", "pdots", "bands"}


def test_restrict_is_for_the_callers_arrays():
    text = ""
    for p in glob.glob(os.path.join(ROOT, "paper_2006_06866_gb300", "csrc", "*.cu*")):
        with open(p) as f:
            text += re.sub(r"//[^\n]*", "", f.read())
    launched = set(re.findall(r"launch_pdl\(\s*(k_\w+)", text))
    assert {"k_scan", "k_trials", "k_prep", "k_main", "k_topk_merge", "k_topk_reduce"} <= launched
    for name in launched:
        m = re.search(r"__global__[^;{]*?\b%s\s*\(([^{]*)\)\s*\{" % name, text)
        assert m, name
        for par in m.group(1).split(","):
            if "__restrict__" in par:
                assert par.split()[-1].lstrip("*") in CALLERS, (name, par.strip())
