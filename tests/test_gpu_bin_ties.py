"""Samples with many points in few cells (ties, rounded data, a range stretched
by outliers), whose weights add up past 32 bits of a cell's fixed-point sum: the
shared-memory histograms of single calls against the additions to global memory
of batches bit for bit (integer sums), and both against the oracle: a weight has
d factors with two roundings of 2^-25 each and d - 1 products, below 2 d 2^-24 in
all, and the count is rounded once."""
import numpy as np
import pytest

from oracle import binning

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,M", [(1, [2]), (1, [700]), (2, [100, 100]), (3, [20, 20, 20]), (4, [10, 9, 8, 11])])
@pytest.mark.parametrize("share", [1.0, 0.5])
def test_ties(d, M, share):
    import torch
    from paper_1511_07482_gb300 import Context
    rng = np.random.default_rng(7 * d + M[0])
    n = 60000
    X = rng.normal(size=(n, d)).clip(-4.9, 4.9)
    X[rng.random(n) < share] *= 1e-7
    X[::5] = X[0]
    lo, hi = np.full(d, -5.0), np.full(d, 5.0)
    x = torch.from_numpy(X).cuda()
    ctx = Context(0)
    ds = [ctx.bin(x, lo, hi, M)] + ctx.bin_many([x, x], [lo, lo], [hi, hi], [M, M])
    got = [o.counts() for o in ds]
    assert all(np.array_equal(g, got[0]) for g in got)
    want = binning.bin_linear(X, lo, hi, M)
    assert np.max(np.abs(got[0] - want)) <= 2.0 ** -24 * (2 * d + 1) * n
    for o in ds:
        o.close()
    ctx.close()
