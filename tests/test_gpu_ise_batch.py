"""The mixture ISE over batches (Eq. 37): one bandwidth and many, one component
and the most that a call takes, grids of a few cells and of many blocks, every
dimension, against the oracle's closed form on the binned sample.

Tolerance: the double sum of the estimate is an FP32 lag sum (1e-5 of its value at
most, the library's stated accuracy), the other two terms are FP64 on FP32 counts
(2e-6); both sums are of the size of the mixture's own square integral."""
import numpy as np
import pytest

from oracle import binning, kde, rules
from paper_1511_07482_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,nH", [([2], 1, 1), ([300], 64, 5), ([3, 2], 2, 40), ([61, 47], 1, 1), ([90, 83], 5, 700),
                                    ([12, 9, 11], 3, 3), ([5, 6, 4, 7], 2, 2)])
def test_batches(M, K, nH):
    from paper_1511_07482_gb300 import Context
    d = len(M)
    w = synthetic.small_case(n=900, d=d, M=M, seed=400 + sum(M) + K, n_candidates=min(nH, 40))
    H = np.stack([w.H[i % len(w.H)] * (1.0 + 0.001 * i) for i in range(nH)])
    rng = np.random.default_rng(K + nH)
    wt = rng.random(K)
    wt /= wt.sum()
    mu = rng.uniform(-1.5, 1.5, (K, d))
    S = np.stack([synthetic.random_spd(rng, d, rng.uniform(0.1, 1.0, d)) for _ in range(K)])
    S = 0.5 * (S + S.transpose(0, 2, 1))
    ctx = Context(0)
    ds = ctx.bin(w.X, w.lo, w.hi, M)
    got = ds.ise_mixture(H, wt, mu, S)
    again = ds.ise_mixture(H[-1:], wt, mu, S)
    c = binning.bin_linear(w.X, w.lo, w.hi, M)
    delta = rules.bin_width(w.lo, w.hi, M)
    scale = kde.mixture_sq_integral(wt, mu, S)
    for i in {0, nH // 2, nH - 1}:
        L = [max(1, v) for v in rules.support_L(rules.lambda_max(2.0 * H[i]), delta, M)]
        want = kde.ise_mixture_binned(c, w.n, np.asarray(w.lo), delta, H[i], wt, mu, S, L)
        tol = 1.2e-5 * max(scale, abs(want) + scale)
        assert abs(got[i] - want) <= tol, (i, got[i], want)
    assert abs(again[0] - got[-1]) <= 1e-12 * max(scale, abs(got[-1]) + scale)
    ds.close()
    ctx.close()
