"""The benchmark's parity block against a stand-in for the library, made of the oracle's own
results, on the CPU: it passes as it is, and a single cell of the searched grid that differs
from what the mode's own fold counts fails it, also where the oracle's bound would let it
pass."""
import sys

import numpy as np
import pytest

from test_host_logic import ROOT

sys.path.insert(0, ROOT)


class Library:
    """gce_ce_grid with `off` added to the cells that are sampled, or to one cell."""
    GCE_OK = 0

    def __init__(self, mode, off):
        self.mode, self.off = mode, off

    class Config:
        def __init__(self, n_phase, n_mag, mode, t0=0.0, overlap=False):
            self.n_phase, self.n_mag, self.mode, self.t0, self.overlap = n_phase, n_mag, mode, t0, overlap

    def _grid(self, cfg, a):
        import oracle
        import torch
        H, _ = oracle.Oracle().ce_grid(a["times"].numpy(), a["mags"].numpy(), a["offsets"], a["periods"].numpy(),
                                       a["pdots"].numpy(), cfg.n_phase, cfg.n_mag, t0=cfg.t0, with_dmin=True,
                                       overlap=cfg.overlap)
        return torch.tensor(H.astype(np.float32))

    def gce_ce_grid(self, h, cfg=None, stream=None, **a):
        H = self._grid(cfg, a)
        if cfg.mode == self.mode:
            worst = H.reshape(H.shape[0], -1).argmax(dim=1)
            if self.mode == "fp64":
                H.view(H.shape[0], -1)[0, worst[0]] += self.off
            else:
                H += self.off
        return H

    def gce_ce_grid_single(self, h, cfg=None, stream=None, **a):
        return self._grid(cfg, a)

    def gce_ce_counts(self, h, cfg=None, cell_curve=None, cell_trial=None, stream=None, **a):
        import oracle
        import torch
        _, _, c = oracle.Oracle().ce_cells(a["times"].numpy(), a["mags"].numpy(), a["offsets"], a["periods"].numpy(),
                                           a["pdots"].numpy(), cfg.n_phase, cfg.n_mag, cell_curve.numpy(),
                                           cell_trial.numpy(), t0=cfg.t0, with_counts=True, overlap=cfg.overlap)
        return torch.tensor(c.astype(np.int32))

    def gce_stream_status(self, h, stream=None):
        return 0


@pytest.mark.parametrize("mode,off,ok", [("none", 0.0, True), ("fp64", 5e-7, False), ("fixed32", 5e-5, False),
                                         ("split32", 5e-5, False)])
def test_searched_grid_is_held_to_its_own_fold(mode, off, ok):
    import bench
    import oracle
    import synth
    oracle.build()
    b = synth.make_config(0)
    ref, dmin = oracle.Oracle().ce_grid(b.times, b.mags, b.offsets, b.periods, b.pdots, b.n_phase, b.n_mag,
                                        with_dmin=True)
    out = bench.parity_block(Library(mode, off), None, "cpu", None, b, ref, dmin, False, n_count_cells=60)
    for m in ("fp64", "split32", "fixed32"):
        assert out[m]["pass"] == (ok or m != mode), out[m]
