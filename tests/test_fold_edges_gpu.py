"""The CE kernel's grid against the entropy of the diagnostic kernel's counts (one
point at a time, no sweeps, no pairing) at the sizes where the hot loop and the
sweeps can go wrong: curve lengths around the staging, pairing and counter-format
edges, every number of trials per thread, one Pdot value and several, plain and
overlapping bins."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# H is float32 (half an ulp below 4: 1.2e-7); the c ln c table adds at most
# 2^-33 per term, 2 (n_mag n_phase + n_phase) terms over N: below 1e-7 here
TOL = 3e-7


def entropy(counts, n):
    c = counts.astype(np.float64)
    ent = lambda x: np.where(x > 1, x * np.log(np.maximum(x, 1)), 0.0)
    return (ent(c.sum(1)).sum(1) - ent(c).sum((1, 2))) / n


def make(lengths, seed, clump=False):
    rng = np.random.default_rng(seed)
    offs = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    t = np.sort(rng.uniform(0, 9.4e7, offs[-1]))
    m = rng.normal(15, 0.1, offs[-1])
    if clump:  # most points in one magnitude bin: one long segment, many short ones
        m = np.where(rng.random(offs[-1]) < 0.8, 15.0 + 1e-3 * rng.random(offs[-1]), 15.0 + rng.random(offs[-1]))
    return t, m, offs


@pytest.mark.parametrize("mode", ["split32", "fixed32", "fp64"])
@pytest.mark.parametrize("shape", [(128, 1, 256, 0), (256, 2, 512, 0), (128, 4, 256, 1)])
@pytest.mark.parametrize("n_pdots", [1, 3])
@pytest.mark.parametrize("bins,overlap", [((15, 10), False), ((50, 7), True), ((2, 1), True)])
def test_grid_is_the_entropy_of_the_counts(mode, shape, n_pdots, bins, overlap):
    import torch

    import paper_2006_06866_gb300 as g
    block, tpt, chunk, rng_ = shape
    if mode == "fp64" and tpt == 4:
        tpt = 2
    lengths = [1, 2, 3, 4, 5, 31, 32, 33, 62, 63, 64, 65, 127, 255, 256, 257, 511, 513, 1023, 1024,
               1025, 2049]
    dev = torch.device("cuda")
    for clump in (False, True):
        t, m, offs = make(lengths, 7, clump)
        periods = np.geomspace(200.0, 5e5, 97)
        pdots = np.linspace(-1e-10, 0.0, n_pdots) if n_pdots > 1 else np.zeros(1)
        d = lambda a: torch.tensor(a, device=dev)
        h = g.Handle(0)
        cfg = g.Config(bins[0], bins[1], mode, overlap=overlap)
        for hint in (1 << e for e in range(1, 13)):
            g.gce_set_tuning(h, cfg, hint, block=block, tpt=tpt, chunk=chunk, slot_range=rng_)
        args = (d(t), d(m), offs, d(periods), d(pdots), cfg)
        H = g.gce_ce_grid(h, *args).cpu().numpy().reshape(len(lengths), -1)
        nt = H.shape[1]
        cc = torch.arange(len(lengths), device=dev).repeat_interleave(nt)
        ct = torch.arange(nt, device=dev).repeat(len(lengths))
        counts = g.gce_ce_counts(h, *args, cell_curve=cc, cell_trial=ct).cpu().numpy()
        assert g.gce_stream_status(h) == g.GCE_OK
        n = np.repeat(np.asarray(lengths), nt) * (2 if overlap else 1)
        want = entropy(counts, n).reshape(H.shape)
        assert np.all(counts.sum((1, 2)) == n)
        err = np.abs(H - want)
        assert err.max() <= TOL, (clump, np.unravel_index(err.argmax(), err.shape), err.max())
        h.close()
