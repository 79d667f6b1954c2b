"""Large FP64 jobs without a tuned shape take four trials per thread, as FIXED32's do: the
grid and the top-k have to be those of one trial per thread bit for bit, inside the coarse
fold's range and beyond it, with trials left over at the grid's end."""
import numpy as np
import pytest

from test_fp64_certified_gpu import job

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["on_edges", "cycles20", "cycles23"])
@pytest.mark.parametrize("n_pdots", [1, 4, 7])
@pytest.mark.parametrize("bins,overlap", [((15, 10), False), ((15, 10), True), ((33, 10), False)])
def test_four_trials_per_thread(kind, n_pdots, bins, overlap):
    import torch

    import paper_2006_06866_gb300 as g
    t, periods, _, t0 = job(kind)
    n_p = 2_000_003 // (4 * n_pdots)  # with four curves 62500 warps of single trials
    periods = np.resize(periods, n_p) * np.linspace(1.0, 1.5, n_p)
    pdots = np.linspace(-1e-12, 0.0, n_pdots) if n_pdots > 1 else np.zeros(1)
    m = np.random.default_rng(5).normal(15, 0.1, t.size)
    cuts = np.array([0, 40, 41, 100, 133])
    d = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    cfg = g.Config(bins[0], bins[1], "fp64", t0=t0, overlap=overlap)
    args = (d(t[:133]), d(m[:133]), cuts, d(periods), d(pdots), cfg)
    got = []
    for tuned in (False, True):
        h = g.Handle(0)
        if tuned:
            for e in range(0, 12):
                g.gce_set_tuning(h, cfg, 1 << e, block=128, tpt=1, chunk=512)
        got.append((g.gce_ce_grid(h, *args), *g.gce_ce_detect(h, *args, k=5)))
        assert g.gce_stream_status(h) == g.GCE_OK
        h.close()
    a, b = got
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    for x, y in zip(a[3:5], b[3:5]):
        assert torch.allclose(x, y, rtol=1e-5, atol=1e-7)
