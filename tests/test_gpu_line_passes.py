"""The autocorrelation's passes at the edges of their line groups: odd numbers
of lines (the last shared transform holds one), padded sizes of every radix,
the shortest axes, every dimension, FP32 (pairs) and FP64, one data set and
many of uneven sizes in one launch.

The library's own counts are read back and their autocorrelation is taken in
FP64, so what is compared is the transform alone: the pairs carry about 44
bits, and an error of a few 2^-44 of a_0 per radix stage (at most 12 stages a
pass, 2 d - 1 passes) stays below 1e-12 a_0, the bound of the other
autocorrelation tests."""
import numpy as np
import pytest

from oracle import functionals as F
from paper_1511_07482_gb300 import DT_F64, FP64, synthetic

pytestmark = pytest.mark.gpu


def _check(ds, A):
    c = ds.counts(DT_F64)
    a = F.autocorr_fft(c)
    lags = [np.arange(0 if k == 0 else -Ak, Ak + 1) % a.shape[k] for k, Ak in enumerate(A)]
    got, want = ds.autocorr(A), a[np.ix_(*lags)].T   # the box has j_0 fastest
    assert got.shape == want.shape
    assert np.max(np.abs(got - want)) <= 1e-12 * float(np.sum(c * c)), (c.shape, A)


@pytest.mark.parametrize("prec", [{}, {"precision": FP64}])
@pytest.mark.parametrize("M,A", [([2], [1]), ([3], [0]), ([101], [100]), ([1000], [37]),
                                 ([2, 2], [1, 1]), ([5, 3], [0, 2]), ([37, 53], [36, 11]), ([64, 61], [0, 60]),
                                 ([300, 7], [24, 0]), ([9, 700], [3, 20]), ([243, 125], [0, 0]),
                                 ([3, 2, 5], [1, 1, 4]), ([21, 13, 34], [4, 12, 5]), ([7, 40, 3], [6, 2, 1]),
                                 ([3, 4, 2, 5], [1, 3, 0, 2]), ([9, 7, 11, 8], [2, 3, 1, 4])])
def test_sizes(M, A, prec):
    from paper_1511_07482_gb300 import Context
    w = synthetic.small_case(n=700, d=len(M), M=M, seed=sum(M) + sum(A))
    ctx = Context(0)
    ds = ctx.bin(w.X, w.lo, w.hi, M, **prec)
    _check(ds, A)
    ds.close()
    ctx.close()


def test_many_uneven():
    """Enough lines in one launch for several a block, with a rest."""
    from paper_1511_07482_gb300 import Context
    rng = np.random.default_rng(8)
    ctx = Context(0)
    ws = [synthetic.small_case(n=400, d=2, M=[int(m) for m in rng.integers(40, 140, 2)], seed=200 + i, n_candidates=2)
          for i in range(60)]
    dss = ctx.bin_many([w.X for w in ws], [w.lo for w in ws], [w.hi for w in ws], [w.M for w in ws])
    ctx.batch_lscv(dss, [w.H for w in ws])
    for ds, w in list(zip(dss, ws))[::7]:
        _check(ds, [3, 2])
    for ds in dss:
        ds.close()
    ctx.close()
