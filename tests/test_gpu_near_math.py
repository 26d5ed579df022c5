"""The near rule's own quotient, logarithm of a ratio and arc tangent against
extended precision, with the bounds their derivations give (units of 2^-52 of the
result): 1 for the quotient, 4 for the two functions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_00864_gb300 import bcfmm
    from paper_2112_00864_gb300.build import build
    build()
    return bcfmm


def scaled(rng, n, lo, hi):
    """Mantissas in [1, 2), edges among them, times 2^lo..2^hi."""
    m = rng.uniform(1.0, 2.0, n)
    m[: n // 8] = 1.0 + rng.integers(0, 4, n // 8) * 2.0 ** -52
    m[n // 8: n // 4] = 2.0 - rng.integers(1, 4, n // 4 - n // 8) * 2.0 ** -52
    rng.shuffle(m)
    return np.ldexp(m, rng.integers(lo, hi + 1, n))


def worst(got, ref):
    return float(np.max(np.abs((got - ref) / ref)) * 2.0 ** 52)


@pytest.mark.parametrize("lo,hi", [(0, 0), (-1, 1), (-40, 40), (-480, 480)])
def test_quotient(bc, lo, hi):
    rng = np.random.default_rng(hi)
    a, b = scaled(rng, 200_000, lo, hi), scaled(rng, 200_000, lo, hi)
    for sa in (1.0, -1.0):
        assert worst(bc.debug_near_math("div", sa * a, b), (sa * a).astype(np.longdouble) / b) <= 1.0


@pytest.mark.parametrize("kind", ["any", "near_one", "near_two", "equal_high_words", "table_points"])
def test_log_of_ratio(bc, kind):
    rng = np.random.default_rng(7)
    n = 200_000
    b = scaled(rng, n, -300, 300)
    if kind == "any":
        r = np.exp(rng.uniform(0, 40, n))
    elif kind == "near_one":
        r = 1.0 + np.exp(rng.uniform(np.log(1e-12), np.log(0.3), n))
    elif kind == "near_two":
        r = 2.0 + rng.choice([-1.0, 1.0], n) * np.exp(rng.uniform(np.log(1e-15), np.log(0.1), n))
    elif kind == "equal_high_words":
        r = 1.0 + rng.integers(1, 1 << 12, n) * 2.0 ** -46
    else:
        r = 1.0 + (rng.integers(0, 32, n) + 0.5 + rng.uniform(-1e-6, 1e-6, n)) / 32.0
    a = np.maximum(b * r, np.nextafter(b, np.inf))
    ref = np.log1p((a.astype(np.longdouble) - b) / b)
    assert worst(bc.debug_near_math("log", a, b), ref) <= 4.0


@pytest.mark.parametrize("kind", ["any", "near_axis", "near_diagonal", "equal_high_words", "table_points"])
def test_atan2(bc, kind):
    rng = np.random.default_rng(11)
    n = 200_000
    x = scaled(rng, n, -300, 300) * rng.choice([-1.0, 1.0], n)
    if kind == "any":
        t = np.exp(rng.uniform(-40, 40, n))
    elif kind == "near_axis":
        t = np.exp(rng.choice([-1.0, 1.0], n) * rng.uniform(3, 100, n))
    elif kind == "near_diagonal":
        t = 1.0 + rng.choice([-1.0, 1.0], n) * np.exp(rng.uniform(np.log(1e-15), np.log(0.1), n))
    elif kind == "equal_high_words":
        t = 1.0 + rng.integers(-(1 << 12), 1 << 12, n) * 2.0 ** -46
    else:
        t = (rng.integers(0, 64, n) + 0.5 + rng.uniform(-1e-6, 1e-6, n)) / 64.0
    y = np.abs(x) * t
    ref = np.arctan2(y.astype(np.longdouble), x.astype(np.longdouble))
    assert worst(bc.debug_near_math("atan", y, x), ref) <= 4.0
    zero = np.zeros(4)
    assert worst(bc.debug_near_math("atan", y[:4], zero), np.arctan2(y[:4].astype(np.longdouble), zero.astype(np.longdouble))) <= 4.0
