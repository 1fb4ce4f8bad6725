"""The grid estimate's tile shapes at their edges (Eq. 1, binned) against the
oracle's shifted sums: axes shorter and longer than a tile, one past its edge,
stencils of several staged chunks and as wide as the grid, every dimension,
host and device outputs.

Tolerance: a value is a sum of non-negative terms c K with FP32 counts (at
most two roundings of 2^-24 of the largest weights, and 2^-33 of a point in
fixed point) and FP32 taps (2^-24), summed to about 2^-44: within 4 x 2^-24 of
the largest value, held to 1e-6 of it."""
import numpy as np
import pytest

from oracle import binning, kde, rules
from paper_1511_07482_gb300 import L_FULL, synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,wide,opts", [
    ([2], 1.0, {}), ([31], 1.0, {}), ([65], 30.0, {}), ([700], 4.0, {}),
    ([2, 3], 1.0, {}), ([8, 16], 1.0, {}), ([9, 17], 4.0, {}), ([33, 31], 1.0, {}), ([32, 65], 9.0, {}),
    ([120, 7], 9.0, {}), ([5, 150], 25.0, {}), ([40, 36], 1.0, {"L_basis": L_FULL}), ([200, 330], 1.0, {}),
    ([5, 4, 3], 1.0, {}), ([9, 34, 33], 4.0, {}), ([6, 7, 40], 9.0, {"L_basis": L_FULL}),
    ([4, 5, 6, 7], 1.0, {}), ([3, 2, 17, 18], 9.0, {})])
def test_tile_edges(M, wide, opts):
    import torch
    from paper_1511_07482_gb300 import Context, load
    w = synthetic.small_case(n=500, d=len(M), M=M, seed=90 + sum(M), n_candidates=1)
    H = w.H[0] * wide
    ctx = Context(0)
    ds = ctx.bin(w.X, w.lo, w.hi, M, **opts)
    got = ds.kde_grid(H)
    dev = torch.empty(M, dtype=torch.float64, device="cuda")
    assert load().kdefft_kde_grid(ds.h, np.ascontiguousarray(H).ctypes.data, dev.data_ptr()) == 0
    assert np.array_equal(dev.cpu().numpy(), got)
    c = binning.bin_linear(w.X, w.lo, w.hi, M)
    delta = rules.bin_width(w.lo, w.hi, M)
    L = [m - 1 for m in M] if opts else [max(1, v) for v in rules.support_L(rules.lambda_max(H), delta, M)]
    want = kde.kde_grid(c, w.n, H, delta, L)
    assert np.max(np.abs(got - want)) <= 1e-6 * np.max(want)
    assert not got[want == 0.0].any()
    ds.close()
    ctx.close()
