"""The persistent form's warp pools at the edges of their ranges: batches of
one event, of a warp, of the device's warps and one more; events with more
dipoles than a pool keeps; every number of gluon kernels in both trial modes;
records that fill up; slices of one cycle.  Every event bitwise the plain
form's.  Requires a GB300."""
import numpy as np
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


def _events(g, ws):
    out = {k: v.cpu().numpy().copy() for k, v in ws.scalars().items()}
    n_max = int(out["n_partons"].max()) if ws.n_events else 0
    live = np.arange(n_max)[:, None] < out["n_partons"][None, :]
    for k, v in {**ws.momenta(), **ws.colours()}.items():
        v = v.cpu().numpy()
        out["r_" + k] = np.where(live, v[..., :n_max, :], 0)
    return out


def _compare(g, p, n, capacity=64, cfg=None, layout=0):
    a, b = g.Workspace(n, capacity), g.Workspace(n, capacity, layout=layout)
    g.generate_me(p, a)
    g.shower(p, a)
    g.generate_me(p, b)
    g.shower_persistent(p, b, cfg)
    torch.cuda.synchronize()
    x, y = _events(g, a), _events(g, b)
    for k in x:
        if k != "valid":
            assert np.array_equal(x[k], y[k]), k
    return x


def test_batch_sizes(g):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = g.make_params(seed=21)
    for n in (1, 2, 31, 32, 33, 65, 16 * sms, 16 * sms + 1, 64 * 16 * sms + 3):
        _compare(g, p, n)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("nf", [1, 2, 3, 4, 5])
def test_kernel_counts(g, nf, mode):
    _compare(g, g.make_params(seed=22, n_flavours=nf, trial_mode=mode), 3001, layout=nf % 3)


@pytest.mark.parametrize("mode", [0, 1])
def test_events_larger_than_the_pool(g, mode):
    """Long showers: many events with more than six dipoles above the cutoff."""
    x = _compare(g, g.make_params(seed=23, sqrt_s=500.0, t_cutoff=0.4, trial_mode=mode), 4001, capacity=128)
    assert (x["n_partons"] > 16).sum() > 100


@pytest.mark.parametrize("period", [1, 5, 64])
def test_full_records_and_cycle_limit(g, period):
    for kw, cap in ((dict(seed=24), 4), (dict(seed=24, max_steps=9), 64)):
        x = _compare(g, g.make_params(**kw), 5003, capacity=cap,
                     cfg={"block_threads": 256, "compact_period": period, "blocks_per_sm": 1})
        assert (x["status"] != g.DONE).any()


def test_slices_of_one_cycle(g):
    """A pool advanced one cycle per launch, its list handed on every time."""
    n = 700
    p = g.make_params(seed=25)
    a, pool = g.Workspace(n, 64), g.Workspace(n, 64)
    g.generate_me(p, a)
    g.shower(p, a)
    g.pool_reset(pool)
    g.pool_admit(p, 3, 0, n, 0, pool, 0)
    for r in range(400):
        g.pool_slice(pool, r, 1, n, shared=p if r % 2 else None)
        if g.pool_progress(pool, r + 1) == 0:
            break
    x, y = _events(g, a), _events(g, pool)
    for k in x:
        assert np.array_equal(x[k], y[k]), k
