"""The observables of events of more than 16 partons (a warp each) at the
edges of their classes and lane counts, isotropic and in two narrow jets,
against the oracle with the observables' parity tolerance; and events with
momenta that are zero, equal or undefined, which must not disturb the others.
Requires a GB300."""
import numpy as np
import pytest

from tests import gpu_harness as H
from tests import synthetic_events as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SQRT_S = 91.2


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2403_08692_gb300 as g
    g.load()
    return g


def _two_jets(rng, n):
    """n massless momenta within about 0.05 of one axis, either way."""
    axis = S.random_rotation(rng)
    e = rng.exponential(size=n) + 0.01
    u = np.concatenate([0.05 * rng.normal(size=(n, 2)), rng.choice([-1.0, 1.0], n)[:, None]], axis=1)
    v = e[:, None] * (u / np.linalg.norm(u, axis=1)[:, None]) @ axis.T
    return np.concatenate([e[:, None], v], axis=1) * (SQRT_S / e.sum())


def _observables(g, events, capacity):
    arrays, counts = S.pack_slot_major(events, capacity)
    ws = g.Workspace(len(events), capacity)
    mom = ws.momenta()
    for c in ("e", "px", "py", "pz"):
        mom[c].copy_(torch.from_numpy(arrays[c]))
    ws.scalars()["n_partons"].copy_(torch.from_numpy(counts))
    ws.scalars()["status"].fill_(g.DONE)
    g.observables(g.make_params(sqrt_s=SQRT_S), ws)
    return ws.obs().cpu().numpy().T


@pytest.mark.parametrize("capacity,sizes", [(32, (16, 17, 31, 32)), (128, (33, 63, 64, 65, 95, 96, 97, 127, 128)),
                                            (255, (17, 128, 129, 160, 191, 193, 254, 255))])
def test_sizes(g, oracle_mod, capacity, sizes):
    rng = np.random.default_rng(capacity)
    events = [f(n) for n in sizes for f in ([lambda n: S.rambo(rng, n, SQRT_S)] * 4 + [lambda n: _two_jets(rng, n)] * 4)]
    got = _observables(g, events, capacity)
    for p, o in zip(events, got):
        want = oracle_mod.event_shapes(p, SQRT_S ** 2)
        assert np.all(np.abs(o - want) <= H.OBS_REL * np.abs(want) + H.OBS_ABS), (len(p), o, want)


def test_degenerate_events_among_others(g, oracle_mod):
    rng = np.random.default_rng(7)
    good = [S.rambo(rng, n, SQRT_S) for n in (20, 40, 70, 100)]
    zero, equal, nan = S.rambo(rng, 40, SQRT_S), S.rambo(rng, 40, SQRT_S), S.rambo(rng, 40, SQRT_S)
    zero[3] = zero[17] = 0.0
    equal[1:] = equal[0]
    nan[5, 1] = np.nan
    got = _observables(g, [good[0], zero, good[1], equal, good[2], nan, good[3]], 128)
    for p, o in zip(good, got[::2]):
        want = oracle_mod.event_shapes(p, SQRT_S ** 2)
        assert np.all(np.abs(o - want) <= H.OBS_REL * np.abs(want) + H.OBS_ABS)
    assert got[3][4] == pytest.approx(0.0, abs=1e-12)  # all along one direction: T = 1


@pytest.mark.parametrize("spread", [1e-4, 1e-6, 1e-7, 1e-8])
def test_thrust_of_nearly_planar_and_narrow_events(g, oracle_mod, spread):
    """Third momenta within the FP32 rounding of many pairs' planes: the thrust
    axis found must still be the longest one."""
    rng = np.random.default_rng(11)
    events = []
    for n in (17, 65, 128, 255):
        for _ in range(3):
            phi = rng.uniform(0.0, 2.0 * np.pi, n)
            flat = np.stack([np.cos(phi), np.sin(phi), spread * rng.normal(size=n)], axis=1)
            narrow = np.array([[0.0, 0.0, 1.0], [0.8, 0.0, -0.6], [-0.8, 0.0, -0.6]])[rng.integers(0, 3, n)]
            for u in (flat, narrow + spread * rng.normal(size=(n, 3))):
                u /= np.linalg.norm(u, axis=1)[:, None]
                e = rng.exponential(size=n) + 0.01
                p = np.concatenate([e[:, None], (e[:, None] * u) @ S.random_rotation(rng).T], axis=1)
                events.append(p * (SQRT_S / e.sum()))
    for p, o in zip(events, _observables(g, events, 255)):
        want = oracle_mod.event_shapes(p, SQRT_S ** 2)[4]
        assert abs(o[4] - want) <= H.OBS_REL * abs(want) + H.OBS_ABS, (len(p), o[4], want)
