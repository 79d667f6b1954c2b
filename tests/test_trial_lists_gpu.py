"""Trial lists: every launch shape with two or four trials per thread covers each trial
once and sums the significance's moments over the same lists, so the whole grid and
(mean, std, rho) are the same bits in every one of them; sizes around the 32- and
512-trial edges of the lists."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_periods,n_pdots", [(1, 1), (31, 1), (33, 1), (255, 1), (257, 1), (511, 1),
                                               (512, 1), (545, 1), (1300, 1), (33, 2), (130, 3),
                                               (300, 5)])
@pytest.mark.parametrize("mode", ["split32", "fixed32", "fp64"])
def test_moments_do_not_depend_on_the_shape(n_periods, n_pdots, mode):
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(1)
    d = lambda a: torch.tensor(a, device="cuda")
    offs = np.array([0, 120, 121, 400])
    t, m = d(np.sort(rng.uniform(0, 9e7, 400))), d(rng.normal(15, 0.1, 400))
    p = d(np.geomspace(300.0, 9000.0, n_periods))
    q = d(np.linspace(-1e-10, 0, n_pdots) if n_pdots > 1 else np.zeros(1))
    k = min(4, n_periods * n_pdots)
    first = None
    for block, tpt in [(256, 2), (64, 2), (128, 2), (512, 2)] + (
            [] if mode == "fp64" else [(64, 4), (128, 4), (256, 4)]):
        h = g.Handle(0)
        cfg = g.Config(15, 10, mode)
        for e in range(10):
            g.gce_set_tuning(h, cfg, 1 << e, block=block, tpt=tpt, chunk=256)
        got = [g.gce_ce_grid(h, t, m, offs, p, q, cfg), *g.gce_ce_detect(h, t, m, offs, p, q, cfg, k)]
        assert g.gce_stream_status(h) == g.GCE_OK
        H = got[0].reshape(3, -1)
        assert torch.isfinite(H).all()
        top = H.sort(dim=1, stable=True)
        assert torch.equal(got[1], top.values[:, :k]) and torch.equal(got[2], top.indices[:, :k])
        first = first or got
        for i, (a, b) in enumerate(zip(first, got)):
            # a Pdot axis: the lists are merged in another order (binary64)
            if n_pdots > 1 and i >= 3:
                torch.testing.assert_close(a, b, rtol=1e-6 if i == 5 else 1e-12, atol=1e-14)
            else:
                assert torch.equal(a, b), (block, tpt, i)
        h.close()
