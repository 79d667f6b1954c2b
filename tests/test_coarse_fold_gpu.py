"""FIXED32 jobs run a coarser fold that leaves the points near a phase-bin edge to
FIXED32's own: the grid has to be the entropy of the diagnostic kernel's counts (which
come from FIXED32's fold on every point), also where every point lies on an edge, at
the limits of the coarse range and beyond it, and in runs of more blocks than the
undecided ones are told apart in."""
import numpy as np
import pytest

from test_fold_edges_gpu import TOL, entropy
from test_fp64_certified_gpu import DAY, job

pytestmark = pytest.mark.gpu


def check(t, m, cuts, periods, pdots, t0, bins, overlap, tpt, mode):
    """The job's grid, its periods repeated until it is large enough for the coarse fold."""
    import torch

    import paper_2006_06866_gb300 as g
    d = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    h = g.Handle(0)
    cfg = g.Config(bins[0], bins[1], mode, t0=t0, overlap=overlap)
    for e in range(1, 14):
        g.gce_set_tuning(h, cfg, 1 << e, block=128, tpt=tpt, chunk=4096)
    args = (d(t), d(m), cuts, d(periods), d(pdots), cfg)
    nt, nc = len(periods) * len(pdots), len(cuts) - 1
    reps = 2_000_000 // (nt * nc) + 1
    big = g.gce_ce_grid(h, args[0], args[1], cuts, args[3].repeat(reps), *args[4:])
    big = big.reshape(nc, len(pdots), reps, len(periods))
    assert torch.equal(big, big[:, :, :1].expand_as(big))
    H = big[:, :, 0].cpu().numpy().reshape(nc, -1)
    cc = torch.arange(nc, device="cuda").repeat_interleave(nt)
    counts = g.gce_ce_counts(h, *args, cell_curve=cc, cell_trial=torch.arange(nt, device="cuda").repeat(nc))
    assert g.gce_stream_status(h) == g.GCE_OK
    counts = counts.cpu().numpy()
    n = np.repeat(np.diff(cuts), nt) * (2 if overlap else 1)
    assert np.all(counts.sum((1, 2)) == n)
    assert np.abs(H - entropy(counts, n).reshape(H.shape)).max() <= TOL
    h.close()


@pytest.mark.parametrize("kind", ["on_edges", "before_t0", "cycles20", "cycles23", "cycles27.9",
                                  "pdot_limit"])
@pytest.mark.parametrize("bins,overlap", [((15, 10), False), ((50, 10), True), ((256, 3), False)])
@pytest.mark.parametrize("tpt", [1, 2, 4])
def test_fixed32_near_the_edges(kind, bins, overlap, tpt):
    t, periods, pdots, t0 = job(kind)
    if kind == "pdot_limit":
        pdots = pdots / 2.0  # |Pdot| tau^2 / P^2 < 2^16 strictly
    m = np.random.default_rng(3).normal(15, 0.1, t.size)
    check(t, m, np.array([0, 1, 40, 300, 700]), periods, pdots, t0, bins, overlap, tpt, "fixed32")


@pytest.mark.parametrize("mode", ["fixed32", "fp64"])
@pytest.mark.parametrize("n_pdots", [1, 2])
@pytest.mark.parametrize("n", [495, 496, 512, 513, 3001])
def test_long_runs_on_edges(mode, n_pdots, n):
    """One magnitude bin: runs around and beyond the 31 blocks with bits of their own."""
    rng = np.random.default_rng(n)
    t = rng.integers(0, 400000, n) * 60.0
    t[::7] += rng.uniform(0, 60, t[::7].size)
    pd = np.linspace(-1e-11, 0, n_pdots) if n_pdots > 1 else np.zeros(1)
    check(t, np.full(n, 15.0), np.array([0, n]), np.array([900.0, 1800.0, 1500.0, 3600.0, 90.0 * 7]),
          pd, 0.0, (15, 1), False, 2, mode)
