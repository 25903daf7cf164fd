"""The FP64 helpers of the kernels against the operations they stand for, over
the whole normal range.

Bounds, in units of the last place of the exact result: the reciprocal's last
multiply-add rounds once (1/2) on an approximation good to 2^-57 (1/16): 0.6;
the quotient multiplies it by the numerator, one rounding more and the first
one's error up to doubled by the change of binade: 1.2 + 0.5 = 1.7.  The root
carries half the rounding of x y (1/2 where x y is at the low end of a binade)
and its own rounding (1/2), the remainder 5 r^3 / 16 of the step adds below 1/16
at r = 2^-19: 1.1; the reciprocal root has one product more inside the step: 1.2."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    return P


def normals(n, lo, hi, seed=1):
    """Random mantissas, exponents in [lo, hi), and the ends of binades."""
    r = np.random.default_rng(seed)
    m = 1.0 + r.integers(0, 1 << 52, n) * 2.0 ** -52
    m[: n // 16] = 1.0 + r.integers(0, 64, n // 16) * 2.0 ** -52
    m[n // 16: n // 8] = 2.0 - r.integers(1, 64, n // 8 - n // 16) * 2.0 ** -52
    return np.ldexp(m, r.integers(lo, hi, n))


def ulps(got, exact):
    """|got - exact| in units of the last place; exact in extended precision."""
    e = exact.astype(np.float64)
    return (np.abs(got.astype(np.longdouble) - exact) / np.spacing(np.abs(e)).astype(np.longdouble)).astype(float).max()


needs_long = pytest.mark.skipif(np.finfo(np.longdouble).nmant < 60, reason="no extended precision on this host")


@needs_long
def test_reciprocal_and_quotient(P):
    x = normals(1 << 20, -1021, 1021) * np.where(np.arange(1 << 20) % 2, 1.0, -1.0)
    assert ulps(P.fp64_math_batch("rcp", x)[:, 0], 1 / x.astype(np.longdouble)) <= 0.6
    x, b = normals(1 << 20, -500, 500, 2), normals(1 << 20, -500, 500, 3)
    assert ulps(P.fp64_math_batch("rcp", x, b)[:, 1], b.astype(np.longdouble) / x) <= 1.7


@needs_long
def test_roots(P):
    x = normals(1 << 20, -1022, 1023)
    s = P.fp64_math_batch("sqrt", x)
    assert ulps(s[:, 0], np.sqrt(x.astype(np.longdouble))) <= 1.1
    assert ulps(s[:, 1], 1 / np.sqrt(x.astype(np.longdouble))) <= 1.2


EDGES = np.array([0.0, -0.0, 5e-324, -5e-324, 2.0 ** -1060, 2.0 ** -1022, -2.0 ** -1022, 2.0 ** -1022 * (1 - 2.0 ** -52), 1.0, -1.0,
                  2.0 ** 1023, np.finfo(float).max, -np.finfo(float).max, np.inf, -np.inf, np.nan, -np.nan])


def test_outside_the_normal_range(P):
    with np.errstate(all="ignore"):
        tiny = np.abs(EDGES) < 2.0 ** -1022
        huge = (np.abs(EDGES) > 2.0 ** 1022) & np.isfinite(EDGES)
        r = P.fp64_math_batch("rcp", EDGES)[:, 0]
        bad = tiny | ~np.isfinite(EDGES)
        assert np.isnan(r[bad]).all() and (r[huge] == 0).all()
        s = P.fp64_math_batch("sqrt", EDGES)
        assert (s[tiny, 0] == 0).all() and (s[tiny, 1] == np.inf).all()
        rest = ~tiny & ((EDGES < 0) | ~np.isfinite(EDGES))
        assert np.isnan(s[rest]).all()


def test_bit_tests(P):
    x = np.concatenate([EDGES, normals(4096, -1022, 1023, 5), -normals(4096, -1022, 1023, 6), normals(4096, -24, -4, 7),
                        -normals(4096, -24, -4, 8), [2.0 ** -10, 2.0 ** -18, -2.0 ** -10, -2.0 ** -18]])
    with np.errstate(invalid="ignore"):
        got = P.fp64_math_batch("below_pow2", x)
        assert np.array_equal(got[:, 0], np.abs(x) < 2.0 ** -10) and np.array_equal(got[:, 1], np.abs(x) < 2.0 ** -18)
        got = P.fp64_math_batch("positive", x)
        assert np.array_equal(got[:, 0], x > 0) and np.array_equal(got[:, 1], (x > 0) & np.isfinite(x))
        got = P.fp64_math_batch("not_below_zero", x)[:, 0]
        assert np.array_equal(got, np.where(x < 0, 0.0, x), equal_nan=True)
        for lo, hi in ((1e7, 1e10), (5e-324, np.inf), (1.0, 1.0)):
            y = np.concatenate([x, [lo, hi, np.nextafter(lo, np.inf), np.nextafter(hi, 0.0)]])
            got = P.fp64_math_batch("between", y, lo, hi)
            assert np.array_equal(got[:, 0], (y > lo) & (y < hi))
            assert np.array_equal(got[:, 1], np.abs(y) < 2.0 ** -1022)


@pytest.mark.parametrize("n", [1, 3, 4, 160, 1023, 1024, (1 << 20) - 1, 1 << 20, (1 << 20) + 3])
def test_interval(P, n):
    r = np.random.default_rng(n)
    k = np.unique(np.concatenate([np.arange(min(n, 64) + 1), np.arange(max(0, n - 64), n + 1), r.integers(0, n + 1, 200)])).astype(float)
    g = np.concatenate([EDGES, k, np.nextafter(k, -np.inf), np.nextafter(k, np.inf), r.uniform(-1, n + 1, 20000),
                        r.uniform(0, 1e-3, 100), [n + 1.0, 2.0 ** 20, 2.0 ** 31, 2.0 ** 33, 1e300]])
    got = P.fp64_math_batch("interval", g, float(n))
    with np.errstate(invalid="ignore"):
        ok = (g >= 0) & (g <= n)
    i = np.where(ok, np.minimum(np.floor(np.where(ok, g, 0.0)), n - 1), -1.0)
    assert np.array_equal(got[:, 0], i)
    assert np.array_equal(got[ok, 1], g[ok] - i[ok])
