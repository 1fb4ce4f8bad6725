"""Groups of kernels in the lag domain against the same kernels one by one: every
form (values, values with gradients, psi_r, both precisions, leave-one-out),
half boxes of one point to several tiles, single bandwidths and batches.

A group and a lone bandwidth take the same terms; what differs is nothing (the
tiles and the order of the sums depend on the item alone), so batches are equal
to single calls bit for bit.  Against the oracle's sums over the library's own
counts (FP64): FP32 kernels within 1e-5 of max(|value|, S / 10), S the sum of
the terms' magnitudes (the library's stated accuracy), FP64 within 1e-11."""
import numpy as np
import pytest

from oracle import functionals as F, selectors as S
from paper_1511_07482_gb300 import DT_F64, FP64, synthetic

pytestmark = pytest.mark.gpu


def _ok(got, want, mag, prec):
    tol = 1e-11 if prec else 1e-5
    assert abs(got - want) <= tol * max(abs(want), mag / 10), (got, want, mag)


@pytest.mark.parametrize("prec", [{}, {"precision": FP64}])
@pytest.mark.parametrize("M,wide", [([2], 1.0), ([40], 1.0), ([900], 60.0), ([2, 2], 1.0), ([9, 12], 1.0),
                                    ([70, 64], 9.0), ([5, 4, 3], 1.0), ([16, 13, 15], 4.0), ([4, 3, 5, 4], 1.0),
                                    ([7, 8, 6, 7], 2.0)])
def test_groups(M, wide, prec):
    from paper_1511_07482_gb300 import Context
    d = len(M)
    w = synthetic.small_case(n=600, d=d, M=M, seed=300 + sum(M), n_candidates=3)
    H, G = np.stack(w.H) * wide, w.G
    ctx = Context(0)
    ds = ctx.bin(w.X, w.lo, w.hi, M, **prec)
    loo = ctx.bin(w.X, w.lo, w.hi, M, exact_loo=1, **prec)
    calls = {"lscv": lambda h: ds.lscv(h, grad=True), "value": lambda h: (ds.lscv(h),),
             "loo": lambda h: loo.lscv(h, grad=True), "scv": lambda h: ds.scv(h, G, grad=True),
             "psi0": lambda h: (ds.psi(h, 0),), "psi2": lambda h: (ds.psi(h, 2),), "psi4": lambda h: (ds.psi(h, 4),)}
    for o in (ds, loo):   # the whole box first: a box that grows between calls is transformed anew
        o.autocorr([m - 1 for m in M])
    got = {k: f(H) for k, f in calls.items()}
    for k, f in calls.items():
        for i in range(len(H)):
            for a, b in zip(got[k], f(H[i:i + 1])):
                assert np.array_equal(a[i], b[0]), (k, i)
    a = F.autocorr_fft(ds.counts(DT_F64))
    delta = (np.asarray(w.hi) - np.asarray(w.lo)) / (np.asarray(M) - 1)
    for i, h in enumerate(H):
        L, _ = ds.plan(0, h)
        ev = lambda t: F.lag_sums(a, w.n, t, delta, L)[0]  # noqa: E731
        mag = lambda t: F.lag_sums(a, w.n, t, delta, L)[1]  # noqa: E731
        sv, sg = S.abs_scales(mag, "lscv", h, w.n)
        v, g = S.lscv(ev, h, w.n, grad=True)
        _ok(got["lscv"][0][i], v, sv, prec)
        _ok(got["value"][0][i], v, sv, prec)
        for p in range(d):
            for q in range(d):
                _ok(got["lscv"][1][i][p, q], g[p, q], sg[p, q], prec)
        for r in (0, 2, 4):
            want = S.psi_vector(ev, h, r)
            for k, al in enumerate(np.ndindex(*([d] * r))):
                alpha = tuple(sum(1 for x in al if x == m) for m in range(d))
                _ok(got[f"psi{r}"][0][i][k], want[k], mag([(1.0, h, alpha)]), prec)
    for o in (ds, loo):
        o.close()
    ctx.close()
