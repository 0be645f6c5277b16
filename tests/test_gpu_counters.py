"""The device counters are those of the last shower call, whichever form ran
before it in the workspace.  Requires a GB300."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2403_08692_gb300 as g
    g.load()
    return g


def test_persistent_form_after_the_plain_form(g):
    n = 60_000  # large enough for the plain form to rebuild its list
    p = g.make_params(seed=81)
    ws = g.Workspace(n, 64)
    g.generate_me(p, ws)
    g.shower(p, ws)
    counters = ws.view("counters", torch.int64, (32,))
    assert int(counters[0]) == n and int(counters[27]) > 0
    for call in (lambda: g.shower_persistent(p, ws), lambda: g.shower(p, ws, g.SHOWER_PERSISTENT)):
        counters[21:28] = 7
        counters[29:] = 7
        g.generate_me(p, ws)
        call()
        torch.cuda.synchronize()
        assert int(counters[0]) == n
        assert not bool(counters[21:28].any()) and not bool(counters[29:].any())
