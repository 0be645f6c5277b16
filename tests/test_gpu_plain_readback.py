"""The plain form's host loop takes no list length that an earlier call
published for its own: calls that allow the most cycles (their sequence
numbers once advanced by 2^32 + 1 each, so that every eighth one's met an
earlier one's in the slots that short calls leave alone), a long one after
seven short ones, against the persistent form.  Requires a GB300."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CAP = 64
MOST = 0x7fffffff
SQRT_S = 91.2


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2403_08692_gb300 as g
    g.load()
    return g


def _batch(g, n, t_cutoff, multi):
    """A batch in its initial state and the parameters its calls take (None:
    its job table, whose calls have no cycle limit)."""
    p = g.make_params(seed=71, sqrt_s=SQRT_S, t_cutoff=t_cutoff, max_steps=MOST)
    ws = g.Workspace(n, CAP)
    if multi:
        g.set_jobs([(p, n - n // 3, 0), (p, n // 3, 9000)], ws)
        p = None
    g.generate_me(p, ws)
    return p, ws


def _launches(g, p, ws):
    rc, launches = g.shower(p, ws)
    assert rc == 0
    return launches


@pytest.mark.parametrize("multi", [True, False], ids=["jobs", "one job"])
def test_lengths_of_earlier_calls(g, multi):
    # a call of 14 .. 20 launches
    cutoff = next(t for t in (100.0, 60.0, 40.0, 25.0, 16.0, 10.0, 6.0, 4.0)
                  if 14 <= _launches(g, *_batch(g, 40, t, multi)) <= 20)
    short = 0.2499 * SQRT_S ** 2  # over at the first cutoff check
    first, shorts = _batch(g, 40, cutoff, multi), [_batch(g, 3, short, multi) for _ in range(7)]
    p, ws = _batch(g, 3000, 1.0, multi)
    q, ref = _batch(g, 3000, 1.0, multi)
    g.shower_persistent(q, ref)
    assert 14 <= _launches(g, *first) <= 20
    assert all(_launches(g, *b) <= 3 for b in shorts)
    _launches(g, p, ws)
    torch.cuda.synchronize()
    ours, theirs = ws.scalars(), ref.scalars()
    assert bool((ours["status"] == g.DONE).all())
    for k in ours:
        assert torch.equal(ours[k], theirs[k]), k
