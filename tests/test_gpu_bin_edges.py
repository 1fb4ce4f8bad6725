"""Binning at the edges of its passes against the oracle (Sec. 4 step 1):
samples around a warp and a block, every dimension, grids with a histogram in
shared memory and without, points on nodes, at the bounds, at signed zeros and
outside, samples that are not 16-byte aligned, one data set and many.

Simple counts are exact.  A linear FP32 weight has at most d FP32 roundings of
its factors, d - 1 of the products and 2^-33 of a point in fixed point; a count
is a sum of weights rounded once: within (2 d + 1) 2^-24 of its largest terms,
held to 2e-6 of the largest count and 2^-24 d n of a point's weight.  FP64
weights: 1e-13, against the oracle's weights at the library's own location
(x - lo) * (1 / delta), which is within two ulps of the oracle's quotient."""
import numpy as np
import pytest

from oracle import binning, rules
from paper_1511_07482_gb300 import BIN_SIMPLE, DT_I32, FP64, OUTSIDE_DROP

pytestmark = pytest.mark.gpu


def _sample(rng, n, d, lo, hi, M):
    X = lo + (hi - lo) * rng.random((n, d))
    delta = (hi - lo) / (np.asarray(M) - 1)
    for i in range(0, n, 3):   # on nodes, halfway, at the bounds
        k = int(rng.integers(d))
        X[i, k] = [lo[k], hi[k], lo[k] + delta[k] * rng.integers(M[k]), lo[k] + delta[k] * (rng.integers(M[k]) + 0.5)][
            int(rng.integers(4))]
    if n > 4:
        X[1] = 0.0
        X[2] = -0.0
        X[3, 0] = hi[0] + 1e-3
        X[4, d - 1] = np.nan
    return X


def _at_reciprocal(X, lo, hi, M, monkeypatch):
    delta = rules.bin_width(lo, hi, M)
    with monkeypatch.context() as m:
        m.setattr(binning, "_coords", lambda X, lo, hi, M: (np.minimum((X - lo) * (1.0 / delta), np.asarray(M) - 1.0), delta))
        return binning.bin_linear(X, lo, hi, M)


@pytest.mark.parametrize("d,M", [(1, [2]), (1, [700]), (1, [40000]), (2, [5, 4]), (2, [100, 122]), (2, [130, 95]),
                                 (3, [4, 3, 2]), (3, [30, 26, 28]), (4, [3, 2, 4, 3]), (4, [13, 9, 12, 11])])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 5000])
def test_edges(d, M, n, monkeypatch):
    import torch
    from paper_1511_07482_gb300 import Context
    rng = np.random.default_rng(1000 * d + n + sum(M))
    lo = np.array([0.0, -1.5, -0.3, 0.0])[:d]
    hi = np.array([1.0, 0.0, 2.7, 0.25])[:d]
    X = np.clip(_sample(rng, n, d, lo, hi, M), None, 5.0)
    flat = torch.zeros(n * d + 1, dtype=torch.float64, device="cuda")
    flat[1:] = torch.from_numpy(X.reshape(-1)).cuda()
    odd = flat[1:].reshape(n, d)   # 8 bytes past an aligned address
    ok = np.all((X >= lo) & (X <= hi), axis=1)
    want = binning.bin_linear(X[ok], lo, hi, M)
    want64 = _at_reciprocal(X[ok], lo, hi, M, monkeypatch)
    tol = 2e-6 * want.max() + 2.0 ** -24 * d
    ctx = Context(0)
    for x in (torch.from_numpy(X).cuda(), odd):
        ds = ctx.bin(x, lo, hi, M, outside_policy=OUTSIDE_DROP)
        got = ds.counts()
        assert ds.info()[2] == n - ok.sum()
        assert np.max(np.abs(got - want)) <= tol
        many = ctx.bin_many([x, X], [lo, lo], [hi, hi], [M, M], outside_policy=OUTSIDE_DROP)
        assert all(np.array_equal(m.counts(), got) and m.info()[2] == n - ok.sum() for m in many)
        d64 = ctx.bin(x, lo, hi, M, outside_policy=OUTSIDE_DROP, precision=FP64)
        assert np.max(np.abs(d64.counts() - want64)) <= 1e-13 * max(n, 1)
        ds1 = ctx.bin(x, lo, hi, M, outside_policy=OUTSIDE_DROP, binning=BIN_SIMPLE)
        assert np.array_equal(ds1.counts(DT_I32), binning.bin_simple(X[ok], lo, hi, M))
        for o in [ds, d64, ds1] + many:
            o.close()
    ctx.close()
