"""The measured workloads of the CE (P, Pdot) search, each one pass through a public entry point.

A case is a dict of plain values:
  entry      grid | topk | detect | detect_bands | host | static: the entry point (gce_ce_<entry>)
  mode       fp64 | split32 | fixed32: the phase fold
  n_curves, n_min, n_max   light curves, and the range of their lengths (log-uniform draws)
  n_periods, p_min, p_max  trial periods (seconds; log-spaced)
  n_pdots, pd_lo           period derivatives, linear on [pd_lo, 0]; one value: Pdot = 0
  n_phase, n_mag, overlap  bins; 50 %-overlapping phase bins
  years      baseline of the nightly cadence
  kind       eclipse | mixed (a third each of eclipses, sinusoids and pure noise)
  k          cells kept per curve (entries other than grid)
  n_bands    filters of multi-filter input
  tuned      the launch shape is fitted to the job once, as a survey pipeline does
"""
import numpy as np
import torch

import paper_2006_06866_gb300 as g

DAY = 86400.0
# exact() takes about 1e-10 s per point-trial; larger cases have none
EXACT_POINT_TRIALS = 2.0e10


def _case(name, entry, mode, n_curves, n, n_periods, p=(300.0, DAY), n_pdots=1, pd_lo=0.0,
          bins=(15, 10), overlap=False, years=3.0, kind="eclipse", k=5, n_bands=0, tuned=False):
    c = dict(entry=entry, mode=mode, n_curves=n_curves, n_min=n[0], n_max=n[1],
             n_periods=n_periods, p_min=p[0], p_max=p[1], n_pdots=n_pdots, pd_lo=pd_lo,
             n_phase=bins[0], n_mag=bins[1], overlap=overlap, years=years, kind=kind, k=k,
             n_bands=n_bands, tuned=tuned)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the plain search of one short light curve, its whole CE grid returned: the
        # smallest call, all latency (100 times over a year, 1000 periods 3-60 min)
        _case("plain_fp64_grid", "grid", "fp64", 1, (100, 100), 1000, p=(180.0, 3600.0), years=1.0),
        # one candidate looked at by hand with the default fold
        _case("one_curve_fixed32", "detect", "fixed32", 1, (811, 811), 50000, p=(180.0, DAY)),
        # a few curves at a time from an alert stream, without device allocations
        _case("alerts_split32_static", "static", "split32", 16, (60, 600), 9973, kind="mixed"),
        # a night's candidates searched from host buffers, copies included
        _case("host_split32", "host", "split32", 200, (701, 701), 30011),
        # the survey batch: equal lengths, a wide period grid, the tuned launch shape
        _case("batch_split32", "topk", "split32", 1000, (1000, 1000), 100000, tuned=True),
        # the same search with bit-exact binary64 counts
        _case("batch_fp64", "detect", "fp64", 100, (1000, 1000), 20000),
        # ragged survey data, 50 to 2000 observations, three kinds of sources
        _case("ragged_split32", "topk", "split32", 10000, (50, 2000), 50000, p=(180.0, DAY),
              kind="mixed", tuned=True),
        # the P-Pdot grid of chirping binaries
        _case("pdot_split32", "topk", "split32", 100, (500, 500), 10000, p=(180.0, 900.0),
              n_pdots=256, pd_lo=-1e-10),
        # P-Pdot candidates confirmed with binary64 counts
        _case("pdot_fp64", "topk", "fp64", 23, (487, 487), 10000, p=(180.0, 900.0), n_pdots=16,
              pd_lo=-1e-10),
        # ten-year baseline, 20 phase bins, uneven lengths, the fixed-point fold
        _case("longbase_fixed32", "topk", "fixed32", 100, (200, 1000), 50000, p=(180.0, 3600.0),
              n_pdots=16, pd_lo=-1e-10, bins=(20, 10), years=10.0),
        # 50 overlapping phase bins, the production setting of the paper
        _case("overlap50_split32", "topk", "split32", 50, (600, 1200), 100000, p=(180.0, DAY),
              n_pdots=4, pd_lo=-1e-10, bins=(50, 10), overlap=True),
        # two filters normalised and searched together
        _case("bands_fixed32", "detect_bands", "fixed32", 300, (300, 900), 20000,
              p=(300.0, 3000.0), n_bands=2),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    entry = rng.choice(["grid", "topk", "detect", "detect_bands", "host", "static"])
    mode = rng.choice(["split32", "split32", "fixed32", "fixed32", "fp64"])
    n_lo = log(50, 1200)
    n = (n_lo, min(2000, n_lo * rng.choice([1, 1, 3, 8])))
    pdot = rng.random() < 0.4
    n_pdots = log(2, 256) if pdot else 1
    overlap = rng.random() < 0.25
    n_phase = rng.choice([50, 50, 30]) if overlap else rng.choice([10, 15, 15, 20, 31])
    n_mag = rng.choice([10, 10, 10, 7, 16])
    n_periods = log(500, 100000)
    n_curves = log(1, 2000)
    p_min = rng.choice([180.0, 300.0])
    p = (p_min, rng.choice([900.0, 3600.0, DAY]))
    # no drawn case costs more than the largest listed one; the static entry's
    # 32 MiB workspace and the grid's output bound those two further
    cap = {"split32": 8e10, "fixed32": 6e10, "fp64": 3e9}[mode] * (0.5 if overlap else 1.0)
    if entry == "static":
        n_periods = min(n_periods, max(500, 200000 // n_pdots))
        while n_periods * n_pdots > 200000:
            n_pdots = max(1, n_pdots // 2)
        n_curves = min(n_curves, 64)
        n_curves = max(1, min(n_curves, int(1.2e7 / (n_periods * n_pdots))))
    if entry == "grid":
        n_curves = max(1, min(n_curves, int(1.0e8 / (n_periods * n_pdots))))
    per_curve = n[1] * n_periods * n_pdots
    if per_curve > cap:
        n_pdots = max(1, int(n_pdots * cap / per_curve))
        per_curve = n[1] * n_periods * n_pdots
    n_curves = max(1, min(n_curves, int(cap / per_curve)))
    return _case(None, entry, mode, n_curves, n, n_periods, p=p, n_pdots=n_pdots,
                 pd_lo=-1e-10 if n_pdots > 1 else 0.0, bins=(n_phase, n_mag), overlap=overlap,
                 years=rng.choice([1.0, 3.0, 3.0, 10.0]), kind=rng.choice(["eclipse", "mixed"]),
                 k=rng.choice([1, 5, 5, 10]),
                 n_bands=rng.choice([2, 3]) if entry == "detect_bands" else 0)


def _lengths(case, seed):
    rng = np.random.default_rng([int(seed), 1])
    lo, hi = case["n_min"], case["n_max"]
    n = np.round(np.exp(rng.uniform(np.log(lo), np.log(hi), size=case["n_curves"])))
    return np.clip(n, lo, hi).astype(np.int64)


def _inputs(case, seed):
    """Times (nightly cadence: 240-night seasons, visits in an 8-hour window, sorted per
    curve), magnitudes, host offsets, periods, Pdots and the filter of each point."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 1000003 + 17)
    n = _lengths(case, seed)
    offsets = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    total, nc = int(offsets[-1]), case["n_curves"]

    def u(size, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(size, generator=gen, device=dev, dtype=torch.float64)

    curve = torch.repeat_interleave(torch.arange(nc, device=dev), torch.tensor(n, device=dev))
    years = max(1, int(round(case["years"])))
    season = torch.floor(u(total, 0, years))
    night = season * 365.0 + torch.floor(u(total, 0, 240))
    t = (night + u(total, 0, 8.0 / 24.0)) * DAY
    # sorted per curve: one sort on (curve, time)
    t = (t + curve * 1e9).sort().values - curve * 1e9
    p0 = torch.exp(u(nc, np.log(case["p_min"]), np.log(case["p_max"])))[curve]
    pd = (-10.0 ** u(nc, -12.0, -10.0))[curve] if case["n_pdots"] > 1 else torch.zeros_like(t)
    cyc = t / p0 - 0.5 * pd * (t / p0) ** 2
    phase = cyc + u(nc)[curve]
    phase = phase - torch.floor(phase)
    depth, width = u(nc, 0.1, 1.0)[curve], u(nc, 0.02, 0.08)[curve]
    signal = depth * (torch.exp(-0.5 * ((phase - 0.25) / width) ** 2) +
                      0.5 * torch.exp(-0.5 * ((phase - 0.75) / width) ** 2))
    if case["kind"] == "mixed":
        cls = torch.arange(nc, device=dev)[curve] % 3
        sine = u(nc, 0.05, 0.5)[curve] * torch.sin(2 * np.pi * phase)
        signal = torch.where(cls == 0, signal, torch.where(cls == 1, sine, torch.zeros_like(sine)))
        sigma = u(nc, 0.01, 0.1)[curve]
    else:
        sigma = 0.02
    noise = torch.randn(total, generator=gen, device=dev, dtype=torch.float64)
    m = 15.0 + signal + sigma * noise
    bands = None
    if case["n_bands"]:
        nb = case["n_bands"]
        b = torch.randint(0, nb, (total,), generator=gen, device=dev)
        m = m + u(nb * nc, -0.5, 0.5)[curve * nb + b]
        bands = b.to(torch.uint8)
    periods = torch.tensor(np.geomspace(case["p_min"], case["p_max"], case["n_periods"]), device=dev)
    pdots = torch.tensor(np.linspace(case["pd_lo"], 0.0, case["n_pdots"]) if case["n_pdots"] > 1
                         else np.zeros(1), device=dev)
    return t.contiguous(), m.contiguous(), offsets, periods, pdots, bands


def prepare(case, seed):
    t, m, offsets, periods, pdots, bands = _inputs(case, seed)
    cfg = g.Config(case["n_phase"], case["n_mag"], case["mode"], overlap=case["overlap"])
    state = dict(case=case, cfg=cfg, offsets=offsets, bands=bands)
    state["handle"] = g.Handle(torch.cuda.current_device()) if case["entry"] != "static" else None
    if case["tuned"]:
        g.gce_autotune_job(state["handle"], t, m, offsets, periods, pdots, cfg)
    if case["entry"] == "host":
        t, m, periods, pdots = (x.cpu().pin_memory() for x in (t, m, periods, pdots))
        state["out_H"] = torch.empty((case["n_curves"], case["k"]), dtype=torch.float32,
                                     pin_memory=True)
        state["out_idx"] = torch.empty((case["n_curves"], case["k"]), dtype=torch.int64,
                                       pin_memory=True)
    state["args"] = (t, m, offsets, periods, pdots)
    torch.cuda.synchronize()
    return state


def run(state):
    case, h, cfg = state["case"], state["handle"], state["cfg"]
    t, m, offsets, periods, pdots = state["args"]
    entry, k = case["entry"], case["k"]
    if entry == "grid":
        return g.gce_ce_grid(h, t, m, offsets, periods, pdots, cfg)
    if entry == "topk":
        return g.gce_ce_topk(h, t, m, offsets, periods, pdots, cfg, k)
    if entry == "detect":
        return g.gce_ce_detect(h, t, m, offsets, periods, pdots, cfg, k)
    if entry == "detect_bands":
        return g.gce_ce_detect_bands(h, t, m, state["bands"], case["n_bands"], offsets, periods,
                                     pdots, cfg, k)
    if entry == "host":
        return g.gce_ce_topk_host(h, t, m, offsets, periods, pdots, cfg, k, out_H=state["out_H"],
                                  out_idx=state["out_idx"])
    return g.gce_ce_topk_static(t, m, offsets, periods, pdots, cfg, k)


def _mean_length(case):
    lo, hi = case["n_min"], case["n_max"]
    return lo if lo == hi else (hi - lo) / np.log(hi / lo)


def work(case):
    """Bytes: the inputs read once, the outputs written once.  Operations: per point-trial
    the cycles, their fraction, the bin and the count (two more with a Pdot term); per
    (phase bin, magnitude bin) cell a c ln c and its sum."""
    trials = case["n_periods"] * case["n_pdots"]
    nc, n = case["n_curves"], _mean_length(case)
    cells = trials * nc
    points = nc * n
    out = 4 * cells if case["entry"] == "grid" else nc * (
        12 * case["k"] + (20 if case["entry"] in ("detect", "detect_bands") else 0))
    ops = cells * (n * (6 if case["n_pdots"] > 1 else 4) + 2 * case["n_phase"] * case["n_mag"])
    return {"bytes": float(points * (17 if case["n_bands"] else 16) +
                           8 * (case["n_periods"] + case["n_pdots"]) + out),
            "flops": float(ops)}


def _band_normalised(m, b, nb):
    v = torch.empty_like(m)
    for i in range(nb):
        x = m[b == i]
        if x.numel() == 0:
            continue
        s = x.sort().values
        med = (s[(s.numel() - 1) // 2] + s[s.numel() // 2]) * 0.5
        sd = x.std(unbiased=False)
        v[b == i] = (x - med) / sd if float(sd) > 0 else torch.zeros_like(x)
    return v


def exact(case, seed):
    trials = case["n_periods"] * case["n_pdots"]
    if _mean_length(case) * case["n_curves"] * trials > EXACT_POINT_TRIALS or case["n_curves"] > 400:
        return None
    t, m, offsets, periods, pdots, bands = _inputs(case, seed)
    dev = t.device
    f = (1.0 / periods).repeat(case["n_pdots"])
    a = 0.5 * pdots.repeat_interleave(case["n_periods"]) * f * f
    np_, nm = case["n_phase"], case["n_mag"]
    width = nm * np_
    lnc = torch.arange(0, 2 * case["n_max"] + 2, device=dev, dtype=torch.float64)
    lnc = torch.where(lnc > 1, lnc * torch.log(lnc.clamp(min=1)), torch.zeros_like(lnc))
    rows = []
    for c in range(case["n_curves"]):
        lo, hi = int(offsets[c]), int(offsets[c + 1])
        tau, mag = t[lo:hi], m[lo:hi]
        if bands is not None:
            mag = _band_normalised(mag, bands[lo:hi], case["n_bands"])
        mn, mx = mag.min(), mag.max()
        mb = torch.zeros_like(mag, dtype=torch.int64) if float(mx) == float(mn) else (
            torch.floor((mag - mn) / (mx - mn) * nm).long().clamp(max=nm - 1))
        H = torch.empty(trials, device=dev, dtype=torch.float64)
        step = max(1, 100_000_000 // (hi - lo))
        for s in range(0, trials, step):
            x = tau * f[s:s + step, None]
            if case["n_pdots"] > 1:
                x -= a[s:s + step, None] * (tau * tau)
            x -= torch.floor(x)
            j = (x.mul_(np_)).to(torch.int32).clamp_(max=np_ - 1)
            ntr = j.shape[0]
            flat = torch.arange(ntr, device=dev, dtype=torch.int32)[:, None] * width
            flat = (flat + mb[None].to(torch.int32) * np_ + j).reshape(-1)
            cnt = torch.zeros(ntr * width, device=dev, dtype=torch.int32)
            cnt.index_add_(0, flat, torch.ones(1, device=dev, dtype=torch.int32).expand(flat.numel()))
            cnt = cnt.reshape(ntr, nm, np_)
            if case["overlap"]:
                cnt = cnt + torch.roll(cnt, -1, dims=2)
            n_eff = (hi - lo) * (2 if case["overlap"] else 1)
            H[s:s + step] = (lnc[cnt.sum(1)].sum(1) - lnc[cnt.long()].sum((1, 2))) / n_eff
        rows.append(H)
    H = torch.stack(rows).clamp(min=0)
    if case["entry"] == "grid":
        return H.reshape(case["n_curves"], case["n_pdots"], case["n_periods"])
    top = H.topk(case["k"], dim=1, largest=False, sorted=True).values
    if case["entry"] in ("detect", "detect_bands"):
        mean, std = H.mean(1), H.std(1, unbiased=False)
        rho = torch.where(std > 0, (mean - top[:, 0]) / std, torch.zeros_like(std))
        return top, None, mean, std, rho
    return top, None
