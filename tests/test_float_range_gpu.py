"""SPLIT32 refuses jobs whose values do not fit in floats, and takes those that just do."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# times up to 1, periods near 0.01, Pdots near 1e-4, in other units of time: x scale
@pytest.mark.parametrize("scale,pdot,ok", [
    (1.0, True, True),
    (1e30, False, True), (1e38, False, True), (4e38, False, False), (1e200, False, False),
    (1e19, True, True), (2e19, True, False), (1e30, True, False),
    (1e-35, False, True), (1e-37, False, False), (1e-300, False, False),
    (1e-15, True, True), (1e-19, True, True), (1e-20, True, False),
])
@pytest.mark.parametrize("n_pdots", [1, 3])
@pytest.mark.parametrize("entry", ["grid", "static"])
def test_values_beyond_float(scale, pdot, ok, n_pdots, entry):
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(1)
    t = rng.uniform(0.25, 1.0, 200) * scale
    t[0] = 1.0 * scale
    d = lambda a: torch.tensor(a, device="cuda")
    pd = np.linspace(2e-4, 1e-4, n_pdots) if pdot else np.zeros(n_pdots)
    args = (d(t), d(rng.normal(15, 0.1, 200)), [0, 200], d(np.linspace(0.01, 0.02, 50) * scale), d(pd),
            g.Config(15, 10, "split32"))
    if entry == "static":
        if ok:
            g.gce_ce_topk_static(*args, 3)
        else:
            with pytest.raises(g.GceError) as e:
                g.gce_ce_topk_static(*args, 3)
            assert e.value.status == g.GCE_ERR_UNSUPPORTED
        return
    h = g.Handle(0)
    H = g.gce_ce_grid(h, *args)
    assert g.gce_stream_status(h) == (g.GCE_OK if ok else g.GCE_ERR_UNSUPPORTED)
    if ok:
        want = g.gce_ce_grid(h, *args[:5], g.Config(15, 10, "fp64"))
        # (a point near an edge may lie in the next bin)
        assert (H - want).abs().median() <= 1e-6 and (H - want).abs().max() <= 0.1
    h.close()


def test_no_point_away_from_the_epoch():
    """tau = 0 everywhere and 1/P beyond float: 0 cycles, but an infinite frequency."""
    import torch

    import paper_2006_06866_gb300 as g
    d = lambda a: torch.tensor(a, device="cuda")
    for p, ok in ((1e-37, True), (1e-40, False), (1e-310, False)):
        h = g.Handle(0)
        args = (d(np.zeros(50)), d(np.arange(50.0)), [0, 50], d(np.full(70, p)), d(np.zeros(1)))
        H = g.gce_ce_grid(h, *args, g.Config(15, 10, "split32"))
        assert g.gce_stream_status(h) == (g.GCE_OK if ok else g.GCE_ERR_UNSUPPORTED)
        if ok:
            assert torch.allclose(H, torch.full_like(H, float(np.log(10.0))))
        h.close()
