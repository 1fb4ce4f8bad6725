"""Binning on axes whose step has no finite reciprocal (a range of a few
denormals, a range past the largest double): t = (x - lo) * (1 / delta) is
then infinite or NaN, and the point belongs to node M - 1, as fmin(t, M - 1)
puts it; simple binning takes the quotient itself.

Every weight is 0 or 1 on these axes, so FP32 and simple counts are exact, and
so are FP64 ones; a regular second axis leaves the rounding of its own weights
(below 2^-24 of a point in FP32, the location's own weights in FP64)."""
import numpy as np
import pytest

from paper_1511_07482_gb300 import BIN_SIMPLE, DT_I32, FP64

pytestmark = pytest.mark.gpu

AXES = [(0.0, 4 * 2e-309, 5), (-3e-310, 7e-310, 40), (0.0, 5e-324, 3), (-1.5e308, 1.5e308, 7), (-1.7e308, 1.7e308, 2)]


def _locate(x, lo, hi, M, simple):
    """Base cell and fraction (simple: node and 0) of the points on one axis."""
    with np.errstate(all="ignore"):
        delta = np.float64(hi - lo) / (M - 1)
        y = x - lo
        t = np.fmin(y / delta if simple else y * (np.float64(1.0) / delta), M - 1.0)   # NaN gives M - 1
    if simple:
        return np.floor(t + 0.5).astype(int), np.zeros(len(x))
    l = np.minimum(np.floor(t), M - 2.0)
    return l.astype(int), t - l


def _counts(X, lo, hi, M, simple=False):
    out = np.zeros(M)
    cells = [_locate(X[:, k], lo[k], hi[k], M[k], simple) for k in range(len(M))]
    for corner in np.ndindex(*([2] * len(M))):
        w = np.ones(len(X))
        for (_, f), b in zip(cells, corner):
            w = w * (f if b else 1.0 - f)
        np.add.at(out, tuple(np.minimum(l + b, m - 1) for (l, _), b, m in zip(cells, corner, M)), w)
    return out


@pytest.mark.parametrize("axis", AXES)
@pytest.mark.parametrize("d", [1, 2])
def test_steps_without_reciprocal(axis, d):
    from paper_1511_07482_gb300 import Context
    rng = np.random.default_rng(4)
    n = 300
    lo, hi, M = np.array([axis[0], -1.0])[:d], np.array([axis[1], 2.0])[:d], [axis[2], 20000][:d]
    X = np.empty((n, d))
    u = rng.random(n)
    X[:, 0] = np.clip((1.0 - u) * lo[0] + u * hi[0], lo[0], hi[0])
    X[:5, 0] = [lo[0], hi[0], 0.0, -0.0, hi[0] / 2]
    if d == 2:
        X[:, 1] = rng.uniform(-1.0, 2.0, n)
    ctx = Context(0)
    want, want1 = _counts(X, lo, hi, M), _counts(X, lo, hi, M, simple=True)
    tol = 0.0 if d == 1 else 2.0 ** -24 * n
    ds = [ctx.bin(X, lo, hi, M)] + ctx.bin_many([X, X], [lo, lo], [hi, hi], [M, M])
    for o in ds:
        assert np.max(np.abs(o.counts() - want)) <= tol
    d64, d1 = ctx.bin(X, lo, hi, M, precision=FP64), ctx.bin(X, lo, hi, M, binning=BIN_SIMPLE)
    assert np.max(np.abs(d64.counts() - want)) <= (0.0 if d == 1 else 1e-13 * n)
    assert np.array_equal(d1.counts(DT_I32), want1)
    for o in ds + [d64, d1]:
        o.close()
    ctx.close()
