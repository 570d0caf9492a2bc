"""The FP64 primitives of the flux kernels (quotient, reciprocal, root; a double as two floats and
back) against IEEE arithmetic: every leading significand, both sides of powers of two, the limits of
the fast exponent range, zeros and non-finite values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIV, RCP, SQRT, SPLIT_JOIN, JOIN = range(5)


def run(op, a, b=None):
    import torch
    from paper_2505_24504_gb300 import jfnk
    a = torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    b = None if b is None else torch.from_numpy(np.ascontiguousarray(b, dtype=np.float64)).cuda()
    out = torch.empty_like(a)
    jfnk.arithmetic(op, a, b, out)
    return out.cpu().numpy()


def ulps(got, ref):
    with np.errstate(all="ignore"):
        return np.where((got == ref) | (np.isnan(got) & np.isnan(ref)), 0.0, abs(got - ref) / np.spacing(abs(ref)))


def leading():
    """Every significand of 24 leading bits, with seeded bits below."""
    m = 1.0 + np.arange(1 << 23) * 2.0 ** -23
    return m + np.random.default_rng(1).integers(0, 1 << 29, m.size) * 2.0 ** -52


def edges():
    """Significands within 64 units in the last place of a power of two, on both sides."""
    j = np.arange(64) * 2.0 ** -52
    return np.concatenate([1.0 + j, 2.0 - j[1:]])


@pytest.mark.parametrize("lo", [False, True])
def test_every_leading_significand(lo):
    """Correct rounding for significands in general position: an approximation of 2^-88 misses it only
    within 2^-35 of a tie, 1e-3 expected of 3e7 values."""
    m = leading() if lo else np.floor(leading() * 2.0 ** 23) * 2.0 ** -23
    assert np.array_equal(run(SQRT, m), np.sqrt(m))
    assert np.array_equal(run(SQRT, 2.0 * m), np.sqrt(2.0 * m))
    a = m[np.random.default_rng(2).permutation(m.size)]
    assert np.array_equal(run(DIV, a, m), a / m)
    # reciprocals: 1 / b lies within 2^-88 of a tie for b a few units below a power of two
    assert ulps(run(RCP, m), 1.0 / m).max() <= 1.0
    assert np.count_nonzero(run(RCP, m) != 1.0 / m) <= 4


def test_powers_of_two_and_exponents():
    """One unit in the last place next to powers of two, where quotients come that close to a tie;
    outside the fast exponent range, at zeros and non-finite values the IEEE operations themselves."""
    s = edges()
    a, b = (x.ravel() for x in np.meshgrid(s, s))
    for ea, eb in ((0, 0), (400, -400), (-400, 400), (400, 400), (-400, -400)):
        x, y = np.ldexp(a, ea), -np.ldexp(b, eb)
        assert ulps(run(DIV, x, y), x / y).max() <= 1.0
        assert ulps(run(RCP, y), 1.0 / y).max() <= 1.0
        assert ulps(run(SQRT, x), np.sqrt(x)).max() <= 1.0
    with np.errstate(all="ignore"):
        v = np.array([0.0, -0.0, 1.0, -3.0, np.inf, -np.inf, np.nan, 5e-324, -2.0 ** -1030, 2.0 ** -410, 2.0 ** 410, 1.7e308])
        x, y = (t.ravel() for t in np.meshgrid(v, v))
        far = (abs(y) < 2.0 ** -400) | ~(abs(y) < 2.0 ** 401) | ((x != 0) & ((abs(x) < 2.0 ** -400) | ~(abs(x) < 2.0 ** 401)))
        got = run(DIV, x, y)
        assert ulps(got, x / y)[far].max() == 0.0 and ulps(got, x / y).max() <= 1.0
        assert ulps(run(RCP, v), 1.0 / v).max() == 0.0
        assert ulps(run(SQRT, v), np.sqrt(v)).max() == 0.0


def test_two_floats():
    """A double as two floats and back keeps 2^-47: the second float takes the last 29 bits to 24
    (2^-48), the sum rounds to the double's last place; on either side of every power of two too."""
    rng = np.random.default_rng(5)
    k = np.arange(1, 53)
    near = np.concatenate([1.0 - 2.0 ** -k, 1.0 + 2.0 ** -k, 1.0 - 2.0 ** -k + 2.0 ** -52, edges()])
    x = np.concatenate([np.ldexp(s * near, e) for e in (-60, -1, 0, 1, 60) for s in (1.0, -1.0)] +
                       [rng.standard_normal(1 << 20) * 2.0 ** rng.integers(-60, 60, 1 << 20)])
    assert (abs(run(SPLIT_JOIN, x) - x) / abs(x)).max() <= 2.0 ** -47
    v = np.array([0.0, np.inf, -np.inf, np.nan, 1e60])
    got = run(SPLIT_JOIN, v)
    assert got[0] == 0.0 and got[1] == np.inf and got[2] == -np.inf and np.isnan(got[3]) and got[4] == np.inf


def test_sum_of_two_floats():
    """(float)h + (float)l to the double's last place (2^-52), the low part of either sign, h also a
    power of two."""
    rng = np.random.default_rng(6)
    h = np.concatenate([np.ldexp(s, e) for e in (-40, 0, 40) for s in (np.ones(4096), rng.uniform(1.0, 2.0, 1 << 18))])
    h = (h * rng.choice([-1.0, 1.0], h.size)).astype(np.float32).astype(np.float64)
    l = (h * rng.uniform(-1.0, 1.0, h.size) * 2.0 ** -rng.integers(24, 50, h.size)).astype(np.float32).astype(np.float64)
    assert (abs(run(JOIN, h, l) - (h + l)) / abs(h)).max() <= 2.0 ** -52
