"""A data set's lags and values do not depend on what shares its launches: alone,
and among many data sets of other sizes in one batch, the same bits.  (FP64 data
sets take whole points: FP64 atomics sum the linear weights in any order.)"""
import numpy as np
import pytest

from paper_1511_07482_gb300 import BIN_SIMPLE, FP64, L_FULL, LSCV, synthetic

pytestmark = pytest.mark.gpu


def _cases(d, M, count, n=800):
    rng = np.random.default_rng(11 * d)
    ws = [synthetic.small_case(n=n, d=d, M=M, seed=50 + d, n_candidates=2)]
    for i in range(count):   # most of them its size, the others around it
        Mi = [int(max(4, m + (i % 5 == 0) * rng.integers(-m // 3, m // 3 + 1))) for m in M]
        ws.append(synthetic.small_case(n=n, d=d, M=Mi, seed=400 + i, n_candidates=2))
    return ws


@pytest.mark.parametrize("prec", [{}, {"precision": FP64, "binning": BIN_SIMPLE}])
@pytest.mark.parametrize("d,M,count", [(2, [128, 128], 60), (2, [64, 61], 90), (2, [200, 180], 40), (3, [30, 26, 28], 12),
                                       (1, [500], 30)])
def test_lags_alone_and_in_a_batch(d, M, count, prec):
    from paper_1511_07482_gb300 import Context
    ws = _cases(d, M, count)
    ctx = Context(0)
    alone = ctx.bin(ws[0].X, ws[0].lo, ws[0].hi, ws[0].M, **prec)
    val, grad = alone.lscv(np.stack(ws[0].H), grad=True)
    L = np.max([alone.plan(LSCV, h)[0] for h in ws[0].H], axis=0)
    lags = alone.autocorr(L)
    for at in (0, 1, len(ws) // 2):   # its place in the batch
        order = ws[1:at + 1] + ws[:1] + ws[at + 1:]
        dss = ctx.bin_many([w.X for w in order], [w.lo for w in order], [w.hi for w in order], [w.M for w in order],
                           **prec)
        v, g = ctx.batch_lscv(dss, [np.stack(w.H) for w in order])
        assert np.array_equal(dss[at].autocorr(L), lags)
        k = sum(len(w.H) for w in order[:at])
        assert np.array_equal(v[k:k + len(val)], val) and np.array_equal(g[k:k + len(val)], grad)
        for ds in dss:
            ds.close()
    alone.close()
    ctx.close()


@pytest.mark.parametrize("prec", [{}, {"precision": FP64, "binning": BIN_SIMPLE}])
def test_values_beside_leave_one_out(prec):
    """One Gaussian (Eq. 10) and two (Eq. 8) a bandwidth in one batch, supports
    of several hundred tiles."""
    from paper_1511_07482_gb300 import Context
    ws = [synthetic.small_case(n=800, d=2, M=[1000, 900 + i], seed=60 + i, n_candidates=12) for i in range(3)]
    ctx = Context(0)
    dss = [ctx.bin(w.X, w.lo, w.hi, w.M, exact_loo=i % 2, L_basis=L_FULL, **prec) for i, w in enumerate(ws)]
    Hs = [np.stack(w.H) * 30.0 for w in ws]
    vals = [ds.lscv(h) for ds, h in zip(dss, Hs)]
    v = ctx.batch_lscv(dss, Hs, grad=False)
    assert np.array_equal(v, np.concatenate(vals))
    for ds in dss:
        ds.close()
    ctx.close()
