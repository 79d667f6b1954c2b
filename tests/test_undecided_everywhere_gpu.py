"""Points that lie at a phase-bin edge in every trial (a time at the epoch, or next to it, or
a cadence that the trial frequencies divide) go where the mode's own fold puts them, alone
and beside others, in every kernel that runs the coarse fold."""
import numpy as np
import pytest

from test_coarse_fold_gpu import check

pytestmark = pytest.mark.gpu

N = 300


def times(kind, rng):
    t = np.sort(rng.uniform(1e3, 9.4e7, N))
    k = {"one": [0], "some": [0, 1, 7, 100, 101, 299], "most": list(range(0, N - 20))}[kind[0]]
    at = {"t0": 0.0, "after": 1e-9, "before": -1e-9}[kind[1]]
    t[k] = at
    return t


@pytest.mark.parametrize("at", ["t0", "after", "before"])
@pytest.mark.parametrize("many", ["one", "some", "most"])
@pytest.mark.parametrize("n_pdots", [1, 3])
@pytest.mark.parametrize("bins,overlap", [((15, 10), False), ((20, 4), True)])
@pytest.mark.parametrize("mode,tpt", [("fixed32", 1), ("fixed32", 4), ("fp64", 2)])
def test_at_the_epoch(at, many, n_pdots, bins, overlap, mode, tpt):
    rng = np.random.default_rng(2)
    t0 = 5.0e8 if at == "t0" else 0.0
    t = np.concatenate([times((many, at), rng) for _ in range(4)]) + t0
    m = rng.normal(15, 0.1, t.size)
    m[::3] = np.round(m[::3], 1)
    pd = np.linspace(-1e-11, 1e-11, n_pdots) if n_pdots > 1 else np.zeros(1)
    check(t, m, N * np.arange(5), np.geomspace(200.0, 5e4, 61), pd, t0, bins, overlap, tpt, mode)


@pytest.mark.parametrize("mode", ["fixed32", "fp64"])
@pytest.mark.parametrize("n_pdots", [1, 16])
def test_epoch_costs_no_more_than_another_time(mode, n_pdots):
    """The same curves with their first time at the epoch: the CE kernel within 5 % (the
    coarse fold runs the same points), and within a rounding error of it within 1.7 (one
    more walk of 16 points and one binary64 trial per curve and warp of trials)."""
    import torch

    import paper_2006_06866_gb300 as g
    d = lambda a: torch.tensor(a, device="cuda")
    rng = np.random.default_rng(4)
    base = np.sort(rng.uniform(1e3, 9.4e7, (100, 600)), axis=1)
    m = d(rng.normal(15, 0.1, base.size))
    p, q = d(np.geomspace(300.0, 3000.0, 20000 if n_pdots == 1 else 5000)), d(np.linspace(-1e-10, 0, n_pdots) * (n_pdots > 1))
    cfg = g.Config(15, 10, mode, time_kernel=True)
    h = g.Handle(0)
    ms = []
    for first in (None, 0.0, 1e-9):
        t = base.copy()
        if first is not None:
            t[:, 0] = first
        t = d(t.ravel())
        ks = []
        for _ in range(8):
            g.gce_ce_topk(h, t, m, 600 * np.arange(101), p, q, cfg, 5)
            ks.append(g.gce_kernel_time(h))
        assert g.gce_stream_status(h) == g.GCE_OK
        ms.append(min(ks))
    h.close()
    assert ms[1] <= 1.05 * ms[0] and ms[2] <= 1.7 * ms[0], ms


@pytest.mark.parametrize("n_periods", [1, 63, 300, 4000])
@pytest.mark.parametrize("n_pdots", [1, 3])
@pytest.mark.parametrize("many", ["one", "some", "most"])
def test_small_calls_at_the_epoch(n_periods, n_pdots, many):
    """Untuned small jobs, whose warps share one trial set, and the static entry."""
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(n_periods)
    t = np.concatenate([times((many, "t0"), rng) for _ in range(2)])
    m = rng.normal(15, 0.1, t.size)
    d = lambda a: torch.tensor(a, device="cuda")
    pd = np.linspace(-1e-11, 1e-11, n_pdots) if n_pdots > 1 else np.zeros(1)
    args = (d(t), d(m), [0, N, 2 * N], d(np.geomspace(200.0, 5e4, n_periods)), d(pd))
    cfg = g.Config(15, 10, "fp64")
    h = g.Handle(0)
    grid = g.gce_ce_grid(h, *args, cfg)
    assert torch.equal(grid, g.gce_ce_grid_single(h, *args, cfg))
    k = min(3, n_periods)
    for x, y in zip(g.gce_ce_topk_static(*args, cfg, k), g.gce_ce_topk(h, *args, cfg, k)):
        assert torch.equal(x, y)
    assert g.gce_stream_status(h) == g.GCE_OK
    h.close()
