"""FP64 jobs run the fixed-point fold where it provably puts a point in the binary64
sequence's bin and the binary64 sequence elsewhere: the grid has to equal the plain
binary64 kernel's (gce_ce_grid_single) bit for bit, also where every point lies on
a phase-bin edge, at the limits of the fixed-point range and beyond it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DAY = 86400.0


def job(kind):
    """times, periods, pdots, t0"""
    rng = np.random.default_rng(11)
    n = 700
    if kind == "on_edges":  # multiples of P / 15 and P / 50, in exact and inexact binary64
        t = rng.integers(0, 400000, n) * 60.0
        return t, np.array([900.0, 1800.0, 1500.0, 3600.0, 3000.0, 0.1 * 900, 1 / 3.0 * 900,
                            7.0 * 900]), np.zeros(1), 0.0
    if kind == "before_t0":
        t = rng.uniform(0, 1000 * DAY, n)
        t[:5] = t[7]  # tau = 0 exactly, five times
        return t, np.geomspace(200.0, DAY, 300), np.linspace(-1e-10, 1e-10, 3), t[7]
    if kind.startswith("cycles"):  # 2^20 .. beyond 2^28 cycles: every shift, then binary64 alone
        t = rng.uniform(0, 1000 * DAY, n)
        p = 1000 * DAY / 2.0 ** float(kind[6:])
        return t, p * np.linspace(1.0, 1.7, 200), np.zeros(1), 0.0
    if kind == "pdot_limit":  # |Pdot| tau^2 / P^2 up to 2^16 cycles
        t = rng.uniform(0, 1000 * DAY, n)
        p = np.linspace(400.0, 900.0, 60)
        top = 2.0 ** 16 * 400.0 ** 2 / (1000 * DAY) ** 2
        return t, p, np.array([-top, -top / 7, 0.0, top / 3, top]), 0.0
    if kind == "pdot_beyond":
        t = rng.uniform(0, 1000 * DAY, n)
        return t, np.linspace(400.0, 900.0, 60), np.array([-1e-3, 0.0, 2e-3]), 0.0
    raise ValueError(kind)


@pytest.mark.parametrize("kind", ["on_edges", "before_t0", "cycles20", "cycles23", "cycles26",
                                  "cycles27.9", "cycles30", "pdot_limit", "pdot_beyond"])
@pytest.mark.parametrize("bins,overlap", [((15, 10), False), ((50, 10), True), ((1, 4), False),
                                          ((256, 3), False)])
@pytest.mark.parametrize("tpt", [1, 2])
def test_equals_plain_binary64(kind, bins, overlap, tpt):
    import torch

    import paper_2006_06866_gb300 as g
    dev = torch.device("cuda")
    t, periods, pdots, t0 = job(kind)
    rng = np.random.default_rng(3)
    cuts = np.array([0, 1, 40, 300, 700])
    m = rng.normal(15, 0.1, t.size)
    d = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    h = g.Handle(0)
    cfg = g.Config(bins[0], bins[1], "fp64", t0=t0, overlap=overlap)
    for e in range(1, 11):
        g.gce_set_tuning(h, cfg, 1 << e, block=128, tpt=tpt, chunk=256)
    args = (d(t), d(m), cuts, d(periods), d(pdots), cfg)
    got = g.gce_ce_grid(h, *args)
    want = g.gce_ce_grid_single(h, *args)
    assert g.gce_stream_status(h) == g.GCE_OK
    assert torch.equal(got, want), float((got - want).abs().max())
    h.close()


def test_static_scratch_without_room_for_the_fixed_point_payload():
    """1.2e6 points: 24 bytes each do not fit the built-in scratch, 8 do."""
    import torch

    import paper_2006_06866_gb300 as g
    dev = torch.device("cuda")
    rng = np.random.default_rng(5)
    offs = np.arange(21, dtype=np.int64) * 60000
    t = torch.tensor(np.sort(rng.uniform(0, 9e7, offs[-1])), device=dev)
    m = torch.tensor(rng.normal(15, 0.1, offs[-1]), device=dev)
    p = torch.tensor(np.geomspace(300.0, 9000.0, 40), device=dev)
    q = torch.zeros(1, dtype=torch.float64, device=dev)
    cfg = g.Config(15, 10, "fp64")
    h = g.Handle(0)
    H, idx = g.gce_ce_topk(h, t, m, offs, p, q, cfg, 3)
    Hs, idxs = g.gce_ce_topk_static(t, m, offs, p, q, cfg, 3)
    assert torch.equal(H, Hs) and torch.equal(idx, idxs)
    h.close()
