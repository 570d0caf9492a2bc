"""The FP64 primitives of the flux kernels against IEEE arithmetic: a double as two floats and back on
both sides of powers of two, zeros and non-finite values."""
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


def edges():
    """Significands within 64 units in the last place of a power of two, on both sides."""
    j = np.arange(64) * 2.0 ** -52
    return np.concatenate([1.0 + j, 2.0 - j[1:]])


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
