"""The units of times and periods are the caller's: FP64 and FIXED32 grids of a job whose
times, periods and Pdots are scaled so that tau^2 leaves binary64's range (tau itself, the
cycles and the Pdot cycles do not)."""
import numpy as np
import pytest

from test_fold_edges_gpu import TOL, entropy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("e", [0, 505, 514])
@pytest.mark.parametrize("n_pdots", [2, 5])
@pytest.mark.parametrize("mode", ["fp64", "fixed32"])
def test_times_whose_squares_overflow(e, n_pdots, mode):
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(e)
    t = np.ldexp(rng.uniform(0.25, 1.0, 300), e)
    m = rng.normal(15, 0.1, 300)
    # 2 to 20 cycles, and up to 100 Pdot cycles: a tau^2 = Pdot f^2 tau^2 / 2
    periods = np.ldexp(np.geomspace(0.05, 0.5, 61), e)
    pdots = np.linspace(-0.5, 0.3, n_pdots)
    d = lambda a: torch.tensor(a, device="cuda")
    h = g.Handle(0)
    cfg = g.Config(15, 10, mode)
    reps = 40000 // periods.size + 1  # enough trials for the coarse fold
    cuts = 300 * np.arange(51)
    args = (d(np.tile(t, 50)), d(np.tile(m, 50)), cuts)
    H = g.gce_ce_grid(h, *args, d(periods).repeat(reps), d(pdots), cfg)
    assert g.gce_stream_status(h) == g.GCE_OK
    H = H.reshape(50, n_pdots, reps, periods.size)
    assert torch.equal(H, H[:1, :, :1].expand_as(H))
    nt = periods.size * n_pdots
    one = (args[0][:300], args[1][:300], [0, 300], d(periods), d(pdots), cfg)
    counts = g.gce_ce_counts(h, *one, cell_curve=torch.zeros(nt, dtype=torch.int64, device="cuda"),
                             cell_trial=torch.arange(nt, device="cuda")).cpu().numpy()
    assert g.gce_stream_status(h) == g.GCE_OK
    got = H[0, :, 0].cpu().numpy().reshape(-1)
    assert np.abs(got - entropy(counts, np.full(nt, 300))).max() <= TOL
    if mode == "fp64":
        assert torch.equal(H[0, :, 0], g.gce_ce_grid_single(h, *one).reshape(n_pdots, -1))
    h.close()
