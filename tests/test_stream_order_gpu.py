"""A handle's calls use one workspace, so each waits for the one before it: on streams that
come and go (a new stream may have a destroyed one's handle value), through every entry
point, and with a call that the caller captures into a graph of its own."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def inputs(n_periods):
    import torch
    rng = np.random.default_rng(8)
    d = lambda a: torch.tensor(a, device="cuda")
    return (d(rng.uniform(0, 1e7, 6000)), d(rng.normal(15, 0.1, 6000)), [0, 900, 2500, 6000],
            d(np.geomspace(300.0, 9000.0, n_periods)), d(np.zeros(1)))


def calls(g, cfg):
    import torch
    bands = (torch.arange(6000, device="cuda") % 3).to(torch.uint8)
    return [lambda h, a: g.gce_ce_grid(h, *a, cfg),
            lambda h, a: g.gce_ce_topk(h, *a, cfg, 5),
            lambda h, a: g.gce_ce_detect(h, *a, cfg, 3),
            lambda h, a: g.gce_ce_detect_bands(h, a[0], a[1], bands, 3, *a[2:], cfg, 3)]


def flat(x):
    return list(x) if isinstance(x, (list, tuple)) else [x]


@pytest.mark.parametrize("mode", ["split32", "fixed32", "fp64"])
@pytest.mark.parametrize("use_graph", [True, False])
def test_streams_that_come_and_go(mode, use_graph):
    import torch

    import paper_2006_06866_gb300 as g
    cfg = g.Config(15, 10, mode, use_graph=use_graph)
    long, short = inputs(60000), inputs(700)
    fns = calls(g, cfg)
    h = g.Handle(0)
    want = [[[x.clone() for x in flat(f(h, a))] for a in (long, short)] for f in fns]
    torch.cuda.synchronize()
    cudart = torch.cuda.cudart()
    got = []
    for rep in range(3):
        for i in range(len(fns)):
            for j, a in enumerate((long, short)):
                v = ctypes.c_ulonglong(0)
                assert int(cudart.cudaStreamCreate(ctypes.addressof(v))) == 0
                s = torch.cuda.ExternalStream(v.value)
                s.wait_stream(torch.cuda.current_stream())
                with torch.cuda.stream(s):
                    got.append((i, j, flat(fns[(i + rep) % len(fns)](h, a)), (i + rep) % len(fns)))
                assert int(cudart.cudaStreamDestroy(v.value)) == 0  # its work goes on
    torch.cuda.synchronize()
    for _, j, x, f in got:
        for u, w in zip(x, want[f][j]):
            assert torch.equal(u, w)
    h.close()


@pytest.mark.parametrize("mode", ["split32", "fp64"])
def test_a_call_in_the_callers_own_capture(mode):
    import torch

    import paper_2006_06866_gb300 as g
    cfg = g.Config(15, 10, mode, use_graph=False)
    args = inputs(3000)
    h = g.Handle(0)
    want = flat(g.gce_ce_detect(h, *args, cfg, 3))  # on another stream than the capture
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="relaxed"):
        out = flat(g.gce_ce_detect(h, *args, cfg, 3))
    for _ in range(2):
        for x in out:
            x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for x, w in zip(out, want):
            assert torch.equal(x, w)
    # the handle goes on, on streams of both kinds
    for use_graph in (True, False):
        cfg.use_graph = use_graph
        for s in (torch.cuda.current_stream(), side):
            with torch.cuda.stream(s):
                again = flat(g.gce_ce_detect(h, *args, cfg, 3))
            torch.cuda.synchronize()
            for x, w in zip(again, want):
                assert torch.equal(x, w)
    assert g.gce_stream_status(h) == g.GCE_OK
    h.close()
