"""Groups of kernels on half boxes of many tiles with a partial last one: tiles of
2048 and 4096 points in FP32 (half boxes past 16 K and 64 K points), 256 in
FP64; values and gradients of LSCV, leave-one-out LSCV and SCV, psi_r, against
the oracle's sums over the library's own counts (FP64), with the bounds of the
other group tests: FP32 1e-5 of max(|value|, S / 10), S the sum of the terms'
magnitudes, FP64 1e-11 of it."""
import numpy as np
import pytest

from oracle import functionals as F, selectors as S
from paper_1511_07482_gb300 import DT_F64, FP64, L_FULL, synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [{}, {"precision": FP64}])
@pytest.mark.parametrize("M", [[131, 150], [40, 37, 35], [9, 11, 8, 10]])
def test_tiles(M, prec):
    from paper_1511_07482_gb300 import Context
    d = len(M)
    w = synthetic.small_case(n=900, d=d, M=M, seed=500 + sum(M), n_candidates=2)
    Hs, G = np.stack(w.H) * 3.0, w.G
    ctx = Context(0)
    ds = ctx.bin(w.X, w.lo, w.hi, M, L_basis=L_FULL, **prec)
    loo = ctx.bin(w.X, w.lo, w.hi, M, L_basis=L_FULL, exact_loo=1, binning=0, **prec)
    lv, lg = ds.lscv(Hs, grad=True)
    ov, og = loo.lscv(Hs, grad=True)
    sv, sg = ds.scv(Hs, G, grad=True)
    psi = {r: ds.psi(Hs, r) for r in (0, 2, 4)}
    tol = 1e-11 if prec else 1e-5
    delta = (np.asarray(w.hi) - np.asarray(w.lo)) / (np.asarray(M) - 1)
    L = [m - 1 for m in M]
    auto = [F.autocorr_fft(x.counts(DT_F64)) for x in (ds, loo)]

    def near(got, want, mag):
        assert np.all(np.abs(np.asarray(got) - want) <= tol * np.maximum(np.abs(want), np.asarray(mag) / 10)), (got, want)

    for i, H in enumerate(Hs):
        ev, mag = [[lambda t, a=a, k=k: F.lag_sums(a, w.n, t, delta, L)[k] for a in auto] for k in (0, 1)]
        for got, want, m in ((lv, lg), S.lscv(ev[0], H, w.n, grad=True), S.abs_scales(mag[0], "lscv", H, w.n)), \
                ((ov, og), S.lscv(ev[1], H, w.n, exact_loo=True, grad=True), S.abs_scales(mag[1], "lscv", H, w.n)), \
                ((sv, sg), S.scv(ev[0], H, G, w.n, grad=True), S.abs_scales(mag[0], "scv", H, w.n, G)):
            near(got[0][i], want[0], m[0])
            near(got[1][i], want[1], m[1])
        for r in psi:
            u = S.psi_unique(ev[0], H, r)
            m = S.psi_unique(mag[0], H, r)
            al = [tuple(sum(1 for x in ix if x == k) for k in range(d)) for ix in np.ndindex(*([d] * r))]
            near(psi[r][i], np.array([u[a] for a in al]), np.array([m[a] for a in al]))
    for o in (ds, loo):
        o.close()
    ctx.close()
