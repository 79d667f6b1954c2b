"""Small jobs run with a CTA's warps sharing one trial set: the grid of a few trials
(which takes that path) equals the same trials' cells of a large job (which does
not), for curve and bin counts around the warps' shares."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["split32", "fixed32", "fp64"])
@pytest.mark.parametrize("bins", [(15, 10), (1, 1), (3, 20), (9, 3), (50, 10)])
@pytest.mark.parametrize("n_pdots", [1, 2, 5])
def test_small_job_equals_large_job(mode, bins, n_pdots):
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(2)
    d = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    lengths = [1, 2, 7, 8, 9, 15, 16, 17, 300, 2047, 5001]
    offs = np.concatenate([[0], np.cumsum(lengths)])
    t, m = d(rng.uniform(0, 9e7, offs[-1])), d(rng.normal(15, 0.1, offs[-1]))
    q = d(np.linspace(-1e-10, 0, n_pdots) if n_pdots > 1 else np.zeros(1))
    big = np.geomspace(250.0, 90000.0, 40000 // n_pdots)
    h = g.Handle(0)
    cfg = g.Config(bins[0], bins[1], mode)
    large = g.gce_ce_grid(h, t, m, offs, d(big), q, cfg)
    for n in (1, 33, 1000 // n_pdots):
        pick = np.linspace(0, big.size - 1, n).astype(np.int64)
        # (SPLIT32 and FIXED32 scale by the job's maxima: keep the shortest period)
        small = g.gce_ce_grid(h, t, m, offs, d(big[pick]), q, cfg)
        assert torch.equal(small, large[:, :, torch.tensor(pick, device="cuda")]), n
        one = slice(int(offs[8]), int(offs[9]))
        H, idx, *mom = g.gce_ce_detect(h, t[one].contiguous(), m[one].contiguous(), [0, 300], d(big[pick]), q, cfg, 1)
        Hs = small[8].reshape(-1)
        assert float(H[0, 0]) == float(Hs.min())
        np.testing.assert_allclose(float(mom[0][0]), float(Hs.double().mean()), rtol=1e-6)
    assert g.gce_stream_status(h) == g.GCE_OK
    h.close()
