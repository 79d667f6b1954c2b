"""The preparation and merge kernels at their edges: curves around the shared-memory
capacities of the per-filter statistics and of the magnitude bins, filters with no,
one and many points, magnitudes on bin edges and ranges beyond binary32; top-k merges
around the keys a thread holds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def host_counts(t, m, n_mag, n_phase, period):
    """binary64 statement of the magnitude bins (first Pdot = 0 fold)"""
    mn, mx = m.min(), m.max()
    i = np.zeros(m.size, np.int64) if mx == mn else np.minimum(
        np.floor((m - mn) / (mx - mn) * n_mag).astype(np.int64), n_mag - 1)
    x = t * (1.0 / period)
    j = np.minimum(np.floor((x - np.floor(x)) * n_phase).astype(np.int64), n_phase - 1)
    c = np.zeros((n_mag, n_phase), np.int64)
    np.add.at(c, (i, j), 1)
    return c


@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 8191, 8193, 20000])
@pytest.mark.parametrize("kind", ["plain", "edges", "tiny", "huge"])
@pytest.mark.parametrize("n_mag", [1, 10, 255])
def test_magnitude_bins(n, kind, n_mag):
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(n)
    t = rng.uniform(0, 1e6, n)
    m = {"plain": rng.normal(15, 0.3, n), "edges": rng.integers(0, n_mag + 1, n) / 8.0,
         "tiny": rng.integers(0, 1000, n) * 1e-40, "huge": rng.normal(0, 1e35, n)}[kind]
    d = lambda a: torch.tensor(a, device="cuda")
    h = g.Handle(0)
    c = g.gce_ce_counts(h, d(t), d(m), [0, n], d(np.array([777.7])), d(np.zeros(1)),
                        g.Config(12, n_mag, "fp64"), d(np.zeros(1, np.int64)), d(np.zeros(1, np.int64)))
    assert g.gce_stream_status(h) == g.GCE_OK
    assert np.array_equal(c[0].cpu().numpy(), host_counts(t, m, n_mag, 12, 777.7))
    h.close()


@pytest.mark.parametrize("n", [1, 33, 4095, 4096, 4097])
@pytest.mark.parametrize("n_bands", [1, 2, 3, 8])
def test_filter_statistics(n, n_bands):
    """gce_ce_grid_bands equals gce_ce_grid on magnitudes normalised in point order here."""
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(n + n_bands)
    t, m = rng.uniform(0, 1e6, n), np.round(rng.normal(15, 0.3, n), 2 if n % 2 else 12)
    b = rng.integers(0, n_bands, n)
    if n > 40:
        b[b == n_bands - 1] = 0  # the last filter: one point, or none of several
        b[n // 2] = n_bands - 1
    v = np.zeros(n)
    for f in range(n_bands):
        x = m[b == f]
        if x.size:
            s = np.sort(x)
            med = s[x.size // 2] if x.size % 2 else (s[x.size // 2 - 1] + s[x.size // 2]) * 0.5
            tot = 0.0
            for y in x:
                tot += y
            mean, ss = tot / x.size, 0.0
            for y in x:
                ss += (y - mean) * (y - mean)
            sd = np.sqrt(ss / x.size)
            v[b == f] = (x - med) / sd if sd > 0 else 0.0
    d = lambda a: torch.tensor(a, device="cuda")
    h = g.Handle(0)
    p, q = d(np.geomspace(300.0, 9000.0, 50)), d(np.zeros(1))
    cfg = g.Config(15, 10, "fp64")
    got = g.gce_ce_grid_bands(h, d(t), d(m), d(b.astype(np.uint8)), n_bands, [0, n], p, q, cfg)
    want = g.gce_ce_grid(h, d(t), d(v), [0, n], p, q, cfg)
    assert g.gce_stream_status(h) == g.GCE_OK
    assert torch.equal(got, want)
    h.close()


@pytest.mark.parametrize("n_periods", [1, 64, 700, 52000, 200000])
@pytest.mark.parametrize("k", [1, 5, 64])
def test_merge(n_periods, k):
    import torch

    import paper_2006_06866_gb300 as g
    k = min(k, n_periods)
    rng = np.random.default_rng(4)
    d = lambda a: torch.tensor(a, device="cuda")
    offs = [0, 40, 75]
    args = (d(rng.uniform(0, 1e7, 75)), d(rng.normal(15, 0.1, 75)), offs,
            d(np.geomspace(300.0, 9000.0, n_periods)), d(np.zeros(1)), g.Config(10, 5, "split32"))
    h = g.Handle(0)
    H, idx, mean, std, rho = g.gce_ce_detect(h, *args, k)
    grid = g.gce_ce_grid(h, *args).reshape(2, -1)
    top = grid.sort(dim=1, stable=True)
    assert torch.equal(H, top.values[:, :k]) and torch.equal(idx, top.indices[:, :k])
    torch.testing.assert_close(mean, grid.double().mean(1), rtol=1e-6, atol=0)
    torch.testing.assert_close(std, grid.double().std(1, unbiased=False), rtol=1e-5, atol=1e-9)
    h.close()


def test_calls_in_flight_with_other_offsets_and_streams():
    """Calls queued without waiting, with the same and other offsets and on two streams,
    give what each gives alone."""
    import torch

    import paper_2006_06866_gb300 as g
    rng = np.random.default_rng(6)
    d = lambda a: torch.tensor(a, device="cuda")
    t, m = d(rng.uniform(0, 1e7, 4000)), d(rng.normal(15, 0.1, 4000))
    p, q = d(np.geomspace(300.0, 9000.0, 3000)), d(np.zeros(1))
    cfg = g.Config(15, 10, "split32")
    cuts = [[0, 900, 4000], [0, 900, 4000], [0, 100, 200, 4000], [0, 2000, 4000], [0, 2000, 4000]]
    want = []
    for c in cuts:
        h = g.Handle(0)
        want.append(g.gce_ce_grid(h, t, m, c, p, q, cfg).clone())
        torch.cuda.synchronize()
        h.close()
    h = g.Handle(0)
    side = [torch.cuda.Stream(), torch.cuda.current_stream()]
    torch.cuda.synchronize()
    got = []
    for rep in range(6):
        for i, c in enumerate(cuts):
            s = side[(rep + i) % 2] if rep > 2 else torch.cuda.current_stream()
            with torch.cuda.stream(s):
                got.append((i, g.gce_ce_grid(h, t, m, c, p, q, cfg)))
    torch.cuda.synchronize()
    for i, x in got:
        assert torch.equal(x, want[i])
    h.close()
