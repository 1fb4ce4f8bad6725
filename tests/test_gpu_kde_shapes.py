"""The grid estimate's tile shapes (which one a grid takes follows from its size
and the number of SMs), each on ragged grids of its own, against the oracle's
shifted sums over the library's own counts.

A value is a sum of non-negative terms c K with exact FP32 counts and taps
rounded once to FP32 (2^-24), summed to about 2^-44, so every value, however
small against the largest, is within 2^-23 of itself, and 2^-140 where taps reach
FP32's smallest numbers (2^-149 a term)."""
import numpy as np
import pytest

from oracle import kde, rules
from paper_1511_07482_gb300 import DT_F64, synthetic

pytestmark = pytest.mark.gpu


def _shape(M, nsm):
    """Nodes computed, padding included but no less than four blocks an SM, times
    the cost of a term: 32 x 32, 32 x 8 split over four warps, 16 x 8."""
    outer = int(np.prod(M[:-2]))

    def cost(tx, ty, per):
        return per * max(-(-M[-1] // tx) * tx * (-(-M[-2] // ty) * ty) * outer, nsm * 4 * tx * ty)
    c = {"wide": cost(32, 32, 1.0), "split": cost(32, 8, 1.1), "narrow": cost(16, 8, 1.4)}
    return min(c, key=c.get)


@pytest.mark.parametrize("M,shape,scale", [
    ([401, 403], "split", 0.06), ([67, 97, 101], "split", 0.04), ([801, 805], "wide", 0.02), ([7, 479, 250], "wide", 0.03),
    ([40, 127, 125], "wide", 0.15), ([3, 14, 127, 125], "wide", 0.2), ([90, 77], "narrow", 0.4)])
def test_shapes(M, shape, scale):
    import torch
    from paper_1511_07482_gb300 import Context
    if _shape(M, torch.cuda.get_device_properties(0).multi_processor_count) != shape:
        pytest.skip("another shape on this number of SMs")
    w = synthetic.small_case(n=4000, d=len(M), M=M, seed=17 + sum(M), n_candidates=1)
    H = w.H[0] * scale
    ctx = Context(0)
    ds = ctx.bin(w.X, w.lo, w.hi, M)
    got, c = ds.kde_grid(H), ds.counts(DT_F64)
    delta = rules.bin_width(w.lo, w.hi, M)
    L = [max(1, v) for v in rules.support_L(rules.lambda_max(H), delta, M)]
    want = kde.kde_grid(c, w.n, H, delta, L)
    assert np.all(np.abs(got - want) <= 2.0 ** -23 * want + 2.0 ** -140)
    ds.close()
    ctx.close()
