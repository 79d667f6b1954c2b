"""Values that overflow binary64 stay inside the arrays: FP64 folds whose cycles do (they have
no phase, and count in bin 0), and magnitudes whose range does."""
import numpy as np
import pytest

from test_fold_edges_gpu import TOL, entropy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("period", [1e-305, 1e-310])
@pytest.mark.parametrize("n", [100, 300])
def test_cycles_beyond_binary64(overlap, period, n):
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(3)
    t, m = rng.uniform(1e5, 1e6, n), rng.normal(15, 0.1, n)
    d = lambda a: torch.tensor(a, device="cuda")
    h = g.Handle(0)
    cfg = g.Config(15, 10, "fp64", overlap=overlap)
    args = (d(t), d(m), [0, n], d(np.full(70, period)), d(np.zeros(1)), cfg)
    cells = torch.arange(70, device="cuda")
    c = g.gce_ce_counts(h, *args, cell_curve=torch.zeros_like(cells), cell_trial=cells).cpu().numpy()
    assert g.gce_stream_status(h) == g.GCE_OK
    phase = c.sum(1)
    assert np.all(phase[:, 0] == n) and np.all(phase[:, 1:-1] == 0)
    assert np.all(phase[:, -1] == (n if overlap else 0))
    want = entropy(c, np.full(70, n * (2 if overlap else 1)))
    single = g.gce_ce_grid_single(h, *args)
    assert torch.equal(single, g.gce_ce_grid(h, *args))
    assert np.abs(single.cpu().numpy().reshape(-1) - want).max() <= TOL
    assert g.gce_stream_status(h) == g.GCE_OK
    h.close()


@pytest.mark.parametrize("mode", ["fp64", "split32", "fixed32"])
def test_magnitude_range_beyond_binary64(mode):
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(4)
    m = rng.choice([-1.7e308, 0.0, 1.7e308], 200)
    d = lambda a: torch.tensor(a, device="cuda")
    h = g.Handle(0)
    cells = torch.arange(60, device="cuda")
    c = g.gce_ce_counts(h, d(rng.uniform(0, 1e6, 200)), d(m), [0, 200], d(np.geomspace(300., 9000., 60)),
                        d(np.zeros(1)), g.Config(15, 10, mode), torch.zeros_like(cells), cells)
    assert g.gce_stream_status(h) == g.GCE_OK
    assert torch.all(c.sum((1, 2)) == 200)
    h.close()
