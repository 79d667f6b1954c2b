"""Tuning does not make a job slower than it is untuned: not the job that was tuned, and not
a job of another size that shares its key."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def setup(mode, nc, n, n_periods, n_pdots):
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(5)
    d = lambda a: torch.tensor(a, device="cuda")
    t = np.sort(rng.uniform(1e3, 9.4e7, (nc, n)), axis=1).ravel()
    pd = np.linspace(-1e-10, 0, n_pdots) if n_pdots > 1 else np.zeros(1)
    return (d(t), d(rng.normal(15, 0.1, nc * n)), n * np.arange(nc + 1),
            d(np.geomspace(300.0, 3000.0, n_periods)), d(pd), g.Config(15, 10, mode, time_kernel=True))


def kernel_ms(h, args):
    import paper_2006_06866_gb300 as g
    ms = []
    for _ in range(12):
        g.gce_ce_topk(h, *args, 5)
        ms.append(g.gce_kernel_time(h))
    assert g.gce_stream_status(h) == g.GCE_OK
    return min(ms)


# runs of one kernel differ by 1 %, and the tuner may take either of two shapes that close; the
# own shapes are 7 to 140 % faster than the tuned ones here
@pytest.mark.parametrize("job", [("fp64", 100, 1000, 20000, 1), ("fp64", 23, 487, 10000, 16),
                                 ("split32", 1, 2000, 1000, 1), ("fixed32", 300, 600, 20000, 1)])
def test_tuned_job(job):
    import paper_2006_06866_gb300 as g
    args = setup(*job)
    h = g.Handle(0)
    before = kernel_ms(h, args)
    H, idx = (x.clone() for x in g.gce_ce_topk(h, *args, 5))
    g.gce_autotune_job(h, *args)
    assert kernel_ms(h, args) <= 1.05 * before
    H2, idx2 = g.gce_ce_topk(h, *args, 5)
    assert (H == H2).all() and (idx == idx2).all()
    h.close()


@pytest.mark.parametrize("synthetic", [False, True])
def test_small_job_after_a_large_one_was_tuned(synthetic):
    import paper_2006_06866_gb300 as g
    large, small = setup("split32", 200, 2000, 20000, 1), setup("split32", 1, 2000, 1000, 1)
    h = g.Handle(0)
    before = kernel_ms(h, small)
    if synthetic:
        g.gce_autotune(h, large[-1], 2000, 20000)
    else:
        g.gce_autotune_job(h, *large)
    assert kernel_ms(h, small) <= 1.1 * before
    # a forced shape is taken at every size
    g.gce_set_tuning(h, small[-1], 2000, block=128, tpt=4, chunk=2048, slot_range=1)
    assert kernel_ms(h, small) > 1.5 * before
    h.close()
