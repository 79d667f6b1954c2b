"""The benchmark's roofline counts no more issue slots per point-trial than the profiled
kernels issue."""
import glob
import os
import re
import sys

from test_host_logic import ROOT

sys.path.insert(0, ROOT)


def test_slots_are_a_lower_bound():
    import bench
    seen = 0
    for path in glob.glob(os.path.join(ROOT, "profiles", "k_main_*.md")):
        with open(path) as f:
            text = f.read()
        mode = re.search(r"k_main_(split32|fixed32|fp64)", os.path.basename(path)).group(1)
        pdot = 1 if "pdot" in os.path.basename(path) else 0
        issued = float(re.search(r"thread-instructions per point-trial \| ([0-9.]+)", text).group(1))
        assert bench.FOLD_SLOTS[mode][pdot] + 2 <= issued, (path, issued)
        seen += 1
    assert seen >= 6
