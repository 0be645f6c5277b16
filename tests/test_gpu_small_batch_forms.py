"""The finalisation kernels' forms for small batches give what the forms for
large ones give, bit for bit: event shapes by 16, 8 or 4 lanes per event and
by one thread, validation by lanes and by threads (on broken records too),
histograms with an observable per warp, the buckets of one block; and a pass
captured in a CUDA graph, where its launches are chained.  Requires a
GB300."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CAP = 64


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2403_08692_gb300 as g
    g.load()
    return g


def _showered(g, p, n, first=0):
    ws = g.Workspace(n, CAP, first)
    g.generate_me(p, ws)
    g.shower_persistent(p, ws)
    return ws


@pytest.fixture(scope="module")
def large(g):
    """A batch large enough for one thread per event, and its results."""
    p = g.make_params(seed=41, sqrt_s=200.0)
    ws = _showered(g, p, 180_001)
    g.validate(p, ws)
    g.observables(p, ws)
    return p, ws


@pytest.mark.parametrize("n", [1, 31, 4096, 4097, 9999, 10_000, 29_999, 30_000, 59_999, 60_000])
def test_event_shapes_and_validation(g, large, n):
    p, big = large
    first = 60_000 if n < 60_000 else 0
    ws = _showered(g, p, n, first)
    g.validate(p, ws)
    g.observables(p, ws)
    assert torch.equal(ws.obs(), big.obs()[:, first:first + n])
    assert torch.equal(ws.scalars()["valid"], big.scalars()["valid"][first:first + n])


def test_validation_of_broken_records(g):
    """The same broken records in a batch validated by threads and in batches
    validated by lanes."""
    p = g.make_params(seed=42)
    n, part = 61_001, 20_333
    ws = _showered(g, p, n)
    mom, col, sc = ws.momenta(), ws.colours(), ws.scalars()
    ev = torch.arange(n, device="cuda")
    pick = lambda k: ev[ev % 11 == k]
    mom["px"][0, pick(0)] += 1e-9
    mom["e"][1, pick(1)] *= -1.0
    mom["pz"][1, pick(2)] = float("nan")
    mom["e"][0, pick(3)] += 1e-6
    mom["e"][1, pick(3)] -= 1e-6
    col["flav"][0, pick(4)] = 7
    col["flav"][0, pick(5)] = 1 + col["flav"][0, pick(5)] % 5
    col["acol"][1, pick(6)] += 1
    col["link"][0, 0, pick(7)] = 255
    col["link"][0, 0, pick(8)] = 0
    sc["n_partons"][pick(9)] -= 1
    g.validate(p, ws)
    bits = sc["valid"].clone()
    assert len(torch.unique(bits)) > 5 and int((bits == 0).sum()) > n // 20
    for first in range(0, n, part):
        m = min(part, n - first)
        sub = g.Workspace(m, CAP)
        for name, (src, dst) in {"mom": (mom, sub.momenta()), "col": (col, sub.colours())}.items():
            for k in dst:
                dst[k].copy_(src[k][..., first:first + m])
        sub.scalars()["n_partons"].copy_(sc["n_partons"][first:first + m])
        g.validate(p, sub)
        assert torch.equal(sub.scalars()["valid"], bits[first:first + m])


def test_histograms(g, large):
    p, big = large
    whole = torch.zeros(g.HIST_FIXED_WORDS, dtype=torch.int64, device="cuda")
    g.histograms_fixed(p, big, whole)
    parts = torch.zeros_like(whole)
    for first in range(0, big.n_events, 29_999):
        ws = _showered(g, p, min(29_999, big.n_events - first), first)
        g.validate(p, ws)
        g.observables(p, ws)
        g.histograms_fixed(p, ws, parts)
    assert torch.equal(whole, parts)


@pytest.mark.parametrize("n,cap", [(3000, CAP), (3000, 160), (70_000, 160)])
def test_pass_in_a_graph(g, n, cap):
    """Chained launches, and every event-shape class."""
    p = g.make_params(seed=43, sqrt_s=200.0, t_cutoff=0.5)
    want = torch.zeros(g.HIST_DOUBLES, dtype=torch.float64).pin_memory()
    assert g.run(p, g.Workspace(n, cap), want, g.SHOWER_PERSISTENT)[0] == 0
    ws, hist = g.Workspace(n, cap), torch.zeros(g.HIST_DOUBLES, dtype=torch.float64, device="cuda")
    stats = torch.zeros(64, dtype=torch.int64, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            g.generate_me(p, ws, side)
            g.shower_persistent(p, ws, None, side)
            g.validate(p, ws, side)
            g.observables(p, ws, side)
            g.histograms(p, ws, hist, side)
            g.reduce_stats(ws, stats, side)
    for _ in range(3):
        hist.zero_()
        ws.buffer.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(hist.cpu(), want)
        assert int(stats[0]) == n
