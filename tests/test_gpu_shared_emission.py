"""Emissions of short lists by four lanes each give the events that a thread
per emission gives: small batches of the plain form against the same events of
a batch whose lists are long, bit for bit.  Requires a GB300."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CAP = 48
LARGE = 120_000


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2403_08692_gb300 as g
    g.load()
    return g


def _shower(g, p, n, first=0, layout=0):
    ws = g.Workspace(n, CAP, first, layout=layout)
    g.generate_me(p, ws)
    g.shower(p, ws)
    return ws


@pytest.fixture(scope="module", params=[0, 1], ids=["per kernel", "per dipole"])
def large(g, request):
    p = g.make_params(seed=61, sqrt_s=200.0, t_cutoff=0.5, trial_mode=request.param)
    return p, _shower(g, p, LARGE)


@pytest.mark.parametrize("n,first,layout", [(1, 5, 0), (7, 100, 1), (8, 0, 2), (9, 77, 0), (257, 3000, 1),
                                            (2433, 9000, 2), (20_001, 60_000, 0)])
def test_events_of_short_lists(g, large, n, first, layout):
    p, big = large
    ws = _shower(g, p, n, first, layout)
    pick = slice(first, first + n)
    ours, theirs = ws.scalars(), big.scalars()
    for k in ours:
        if k != "valid":
            assert torch.equal(ours[k], theirs[k][pick]), k
    live = torch.arange(CAP, device="cuda")[:, None] < ours["n_partons"][None, :]
    ours, theirs = {**ws.momenta(), **ws.colours()}, {**big.momenta(), **big.colours()}
    for k in ours:
        assert torch.equal(ours[k][..., live], theirs[k][..., pick][..., live]), k
