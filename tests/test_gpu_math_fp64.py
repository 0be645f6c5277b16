"""The FP64 functions of the splitting kinematics and the dipole cache on the
GPU, against values rounded from extended precision: the errors their
analyses bound (in ulps of the result), over the ranges the shower takes them
in and up to the ends of their own ranges, and the library's values beyond."""
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


def _on_device(g, op, x):
    return g.math_fp64_device(op, torch.from_numpy(np.ascontiguousarray(x)).cuda()).cpu().numpy()


def _two_product(a, b):
    """a b = p + e exactly (Dekker's product on Veltkamp's halves)."""
    split = lambda v: (lambda c: (c - (c - v), v - (c - (c - v))))(134217729.0 * v)
    p = a * b
    (ah, al), (bh, bl) = split(a), split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _ulps(y, residual):
    """The error in ulps of y given (y - exact)."""
    return np.abs(residual) / np.spacing(np.abs(y))


POSITIVE = [("shower", -3.0, 5.0), ("wide", -36.0, 36.0)]


@pytest.mark.parametrize("name,lo,hi", POSITIVE)
def test_reciprocal_and_division(g, name, lo, hi):
    rng = np.random.default_rng(1)
    x = 10.0 ** rng.uniform(lo, hi, 400_000)
    for op, a in (("rcp", 1.0), ("three_over", 3.0)):
        y = _on_device(g, op, x)
        p, e = _two_product(y, x)  # y - a/x = (y x - a) / x, y x exact in two parts
        assert _ulps(y, ((p - a) + e) / x).max() <= 0.52


@pytest.mark.parametrize("name,lo,hi", POSITIVE)
def test_square_roots(g, name, lo, hi):
    rng = np.random.default_rng(2)
    x = 10.0 ** rng.uniform(lo, hi, 400_000)
    y = _on_device(g, "sqrt", x)
    p, e = _two_product(y, y)  # y - sqrt(x) = (y^2 - x) / (2 y) to second order
    assert _ulps(y, ((p - x) + e) / (2.0 * y)).max() <= 1.1
    y = _on_device(g, "rsqrt", x)
    p, e = _two_product(y, y)  # y - x^-1/2 = (x y^2 - 1) y / 2
    q, f = _two_product(p, x)
    assert _ulps(y, (((q - 1.0) + f) + e * x) * y / 2.0).max() <= 0.52


@pytest.mark.parametrize("name,lo,hi", POSITIVE)
def test_square_root_is_as_close_as_the_division(g, name, lo, hi):
    """Half an ulp of the last rounding, and the dropped terms: the low part of
    x y0 is below 2^-53 of the root and its own rounding, with that of the
    correction (2^-21 of the root), below 2^-73."""
    rng = np.random.default_rng(6)
    x = 10.0 ** rng.uniform(lo, hi, 400_000)
    y = _on_device(g, "sqrt", x)
    p, e = _two_product(y, y)
    assert _ulps(y, ((p - x) + e) / (2.0 * y)).max() <= 0.52


def _decimal_check(fn, xs, ys):
    """Largest error in ulps of ys against 40-digit values of fn at xs."""
    from decimal import Decimal, getcontext
    getcontext().prec = 40
    worst = 0.0
    for x, y in zip(xs, ys):
        d = Decimal(float(y)) - fn(Decimal(float(x)))
        worst = max(worst, abs(float(d)) / float(np.spacing(abs(float(y)))))
    return worst


@pytest.mark.parametrize("lo,hi", [(-1.0, 11.0), (-0.02, 0.02), (-599.0, 599.0)])
def test_exponential(g, lo, hi):
    rng = np.random.default_rng(3)
    x = np.concatenate([rng.uniform(lo, hi, 4_000), [0.0, -0.0]])
    y = _on_device(g, "exp", x)
    assert _decimal_check(lambda d: d.exp(), x, y) <= 0.56


@pytest.mark.parametrize("lo,hi", [(-12.0, 0.0), (-0.02, 0.0), (-1e-6, 0.0), (-599.0, 0.0)])
def test_expm1_of_negative(g, lo, hi):
    rng = np.random.default_rng(4)
    x = rng.uniform(lo, hi, 4_000)
    y = _on_device(g, "expm1", x)
    from decimal import Decimal
    assert _decimal_check(lambda d: d.exp() - Decimal(1), x, y) <= 1.6
    assert _on_device(g, "expm1", np.array([0.0]))[0] == 0.0


def _sin_cos(u):
    """40-digit sine and cosine of 2 pi u by their Taylor series."""
    from decimal import Decimal
    pi = Decimal("3.141592653589793238462643383279502884197169399375105820974944592307816406286")
    x = 2 * pi * (u - (u > Decimal("0.5")))
    s, c, term, k = Decimal(0), Decimal(0), Decimal(1), 0
    while abs(term) > Decimal(10) ** -38 or k < 4:
        if k % 2:
            s += term if k % 4 == 1 else -term
        else:
            c += term if k % 4 == 0 else -term
        k += 1
        term = term * x / k
    return s, c


def test_circle(g):
    rng = np.random.default_rng(5)
    m = np.concatenate([rng.integers(0, 1 << 52, 3_000), [0, 1, (1 << 52) - 1, 1 << 51, 1 << 50, 3 << 50],
                        (np.arange(65) << 46).clip(0, (1 << 52) - 1), ((2 * np.arange(64) + 1) << 45)])
    u = (2.0 * m.astype(np.float64) + 1.0) * 2.0 ** -53
    s, c = _on_device(g, "sin_2pi", u), _on_device(g, "cos_2pi", u)
    assert _decimal_check(lambda d: _sin_cos(d)[0], u, s) <= 1.2
    assert _decimal_check(lambda d: _sin_cos(d)[1], u, c) <= 1.2


def test_outside_the_ranges(g):
    x = np.array([0.0, -0.0, 5e-324, 1e-300, 2.0 ** -121, 2.0 ** 121, 1e300, np.inf, np.nan, -4.0])
    with np.errstate(all="ignore"):
        for op, want in (("rcp", 1.0 / x), ("sqrt", np.sqrt(x)), ("rsqrt", 1.0 / np.sqrt(x)),
                         ("exp", np.exp(x)), ("expm1", np.expm1(-np.abs(x)))):
            got = _on_device(g, op, -np.abs(x) if op == "expm1" else x)
            same = (np.isnan(got) & np.isnan(want)) | (got == want) | (np.abs(got - want) <= 2e-16 * np.abs(want))
            assert np.all(same), (op, x[~same], got[~same], want[~same])
