"""What this library is used for, as cases that can be timed and compared.

A case is a dict of plain values; its "kind" says which call of the public
interface it stands for:

  analysis   one small data set from the sample to psi_4 and LSCV at one
             bandwidth: bin, psi, lscv with its gradient (latency and launches)
  select     the selection itself (Eq. 9): bin, then LSCV and SCV minimised
             over full bandwidths from several starts
  objective  a data set that is already binned, evaluated at a batch of
             candidate bandwidths with gradients (what an optimiser or a
             cross-validation loop of the user's own does)
  psi        bin and all partial derivatives of one order at many candidates
  many       many data sets of uneven sizes binned and evaluated in one call
  plugin     bin and the plug-in objective with gradients for a batch of
             candidates, and its eta_{0,2} functional (fourth order)
  kde        the binned density estimate at every grid node
  ise        a simulation study: the integrated squared error of the estimate
             against the normal mixture that the sample was drawn from
  autograd   psi_r and LSCV as differentiable torch functions of H, forward
             and backward
  bin        a large sample onto its grid, and the counts

Samples are draws of normal mixtures with full covariances (random rotations,
eigenvalues in [0.1, 1], means in [-2, 2]^d), the grid covers the sample and
three bandwidths, and candidates lie around the normal-scale bandwidth with
eigenvalues a factor 1/4 to 4 of it.

A data set in FP32 mode is evaluated in FP32 arithmetic, and what it returns
holds about seven digits: a program that chooses that mode keeps the results
as FP32.  Results of FP64 data sets stay FP64.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1511_07482_gb300 import (BIN_LINEAR, BIN_SIMPLE, DT_F32, DT_F64, DT_I32, FP32, FP64, LSCV, P_FIXED, SCV,
                                    Context, load)
from paper_1511_07482_gb300 import autograd as ag

TAU = 3.7


# ------------------------------------------------------------------ the cases
def _case(kind, d, n, M, nH=1, prec="fp32", **more):
    M = [M] * d if isinstance(M, int) else list(M)
    c = {"kind": kind, "d": d, "n": n, "nH": nH, "prec": prec}
    c.update({f"M{k}": M[k] for k in range(d)})
    c.update(more)
    return c


def listed():
    named = [
        # the plain method on a textbook-sized sample: nothing but latency
        ("analysis_2d_n1000", _case("analysis", 2, 1000, 100)),
        # the selector as it is meant to be used: a hundred thousand points,
        # a 256 x 256 grid, both criteria, sixteen starts each
        ("select_2d_n1e5", _case("select", 2, 100_000, 256, nstarts=16)),
        # many candidates on one binned data set
        ("lscv_2d_h256", _case("objective", 2, 100_000, 256, nH=256, method="lscv")),
        # the same in FP64 mode, where an optimiser needs differences of values
        ("scv_2d_fp64_h16", _case("objective", 2, 100_000, 256, nH=16, prec="fp64", method="scv")),
        # an odd-sized three-dimensional grid and a handful of candidates
        ("scv_3d_ragged_h5", _case("objective", 3, 37_411, (61, 97, 45), nH=5, method="scv")),
        # fourth-order functionals of a large three-dimensional sample
        ("psi4_3d_n1e6_h256", _case("psi", 3, 1_000_000, 128, nH=256, r=4)),
        # hundreds of small data sets at once, n from 1e3 to 1e5
        ("many_2d_512x16", _case("many", 2, 100_000, 256, nH=16, sets=512)),
        # the plug-in selector's functionals in four dimensions
        ("plugin_4d_n1e6", _case("plugin", 4, 1_000_000, 48, nH=8, P=96)),
        # the estimate itself, at every node of a three-dimensional grid
        ("kde_3d_n1e6", _case("kde", 3, 1_000_000, 128)),
        # one replicate of a simulation study over a path of bandwidths
        ("ise_2d_n2000_h32", _case("ise", 2, 2000, 101, nH=32)),
        # bandwidths learned by gradient descent inside a torch program
        ("autograd_2d_h16", _case("autograd", 2, 20_000, 128, nH=16, r=2)),
        # a large sample onto a fine grid
        ("bin_2d_n1e7", _case("bin", 2, 10_000_000, 512)),
    ]
    return [dict(c, name=n) for n, c in named]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["analysis", "select", "objective", "objective", "psi", "many", "plugin", "kde", "ise",
                       "autograd", "bin", "bin"])
    side = {1: (64, 1500), 2: (24, 400), 3: (16, 128), 4: (10, 40)}

    def grid(d, hi=None):
        a, b = side[d]
        return [_log(rng, a, min(b, hi or b)) for _ in range(d)]

    if kind == "analysis":
        d = rng.choice([1, 2, 2, 3])
        return _case(kind, d, _log(rng, 100, 5000), grid(d, 200 if d < 3 else 48), prec=rng.choice(["fp32", "fp64"]))
    if kind == "select":
        return _case(kind, 2, _log(rng, 1000, 100_000), grid(2, 256), nstarts=rng.randint(3, 16))
    if kind == "objective":
        d = rng.choice([1, 2, 2, 3, 3])
        prec = rng.choice(["fp32", "fp32", "fp64"])
        top = {1: 512, 2: 512, 3: 64}[d] if prec == "fp32" else {1: 256, 2: 64, 3: 3}[d]
        return _case(kind, d, _log(rng, 1000, 300_000), grid(d, None if prec == "fp32" or d < 3 else 64),
                     nH=_log(rng, 1, top), prec=prec, method=rng.choice(["lscv", "scv"]))
    if kind == "psi":
        d = rng.choice([2, 3, 3])
        return _case(kind, d, _log(rng, 10_000, 1_000_000), grid(d), nH=_log(rng, 1, 256), r=rng.choice([0, 2, 4, 4]))
    if kind == "many":
        return _case(kind, 2, _log(rng, 2000, 100_000), rng.randint(24, 256), nH=rng.randint(1, 16),
                     sets=_log(rng, 2, 400))
    if kind == "plugin":
        d = rng.choice([2, 3, 4, 4])
        return _case(kind, d, _log(rng, 10_000, 1_000_000), grid(d), nH=_log(rng, 1, 16), P=0)
    if kind == "kde":
        most = work(_case("kde", 3, 1_000_000, 128))["flops"]
        while True:   # small samples have wide stencils: none that costs more than the listed one
            d = rng.choice([1, 2, 3, 3])
            c = _case(kind, d, _log(rng, 1000, 1_000_000), grid(d))
            if work(c)["flops"] <= 0.7 * most:
                return c
    if kind == "ise":
        d = rng.choice([1, 2, 2])
        return _case(kind, d, _log(rng, 300, 10_000), grid(d, 200), nH=_log(rng, 1, 64))
    if kind == "autograd":
        d = rng.choice([1, 2, 2, 3])
        return _case(kind, d, _log(rng, 1000, 100_000), grid(d, 200 if d < 3 else 48), nH=_log(rng, 1, 64),
                     r=rng.choice([0, 2]))
    d = rng.choice([1, 2, 3, 4])
    return _case(kind, d, _log(rng, 100_000, 8_000_000), grid(d), prec=rng.choice(["fp32", "fp32", "fp64"]),
                 rule=rng.choice(["linear", "linear", "simple"]))


def _M(case):
    return [case[f"M{k}"] for k in range(case["d"])]


# ------------------------------------------------------------------ inputs
_CTX = None


def _ctx():
    """The one context that a program keeps."""
    global _CTX
    if _CTX is None:
        _CTX = Context(0)
    return _CTX


def _rotation(rng, d):
    Q, R = np.linalg.qr(rng.standard_normal((d, d)))
    return Q * np.sign(np.diag(R))[None, :]


def _sample(rng, gen, n, d, K):
    """n points of a K-component normal mixture on the GPU, and the mixture."""
    w = 0.15 + rng.random(K)
    w /= w.sum()
    mu = rng.uniform(-2.0, 2.0, size=(K, d))
    S = np.empty((K, d, d))
    for k in range(K):
        Q = _rotation(rng, d)
        S[k] = Q @ np.diag(rng.uniform(0.1, 1.0, d)) @ Q.T
        S[k] = 0.5 * (S[k] + S[k].T)
    lab = torch.searchsorted(torch.tensor(np.cumsum(w)[:-1], device="cuda"),
                             torch.rand(n, generator=gen, device="cuda", dtype=torch.float64))
    z = torch.randn(n, d, generator=gen, device="cuda", dtype=torch.float64)
    chol = torch.tensor(np.linalg.cholesky(S), device="cuda")
    X = torch.tensor(mu, device="cuda")[lab]
    for k in range(K):   # n x d products, a component at a time (no n x d x d copy)
        X += torch.where((lab == k)[:, None], z @ chol[k].T, torch.zeros((), dtype=torch.float64, device="cuda"))
    return X.contiguous(), (w, mu, S)


def _scale(X):
    """The normal-scale bandwidth and the range of the sample."""
    n, d = X.shape
    S = torch.cov(X.T).reshape(d, d) if n > 1 else torch.eye(d, dtype=torch.float64, device=X.device)
    back = torch.cat([S.reshape(-1), X.amin(0), X.amax(0)]).cpu().numpy()
    H = (4.0 / (d + 2.0)) ** (2.0 / (d + 4.0)) * n ** (-2.0 / (d + 4.0)) * back[:d * d].reshape(d, d)
    H = 0.5 * (H + H.T)
    pad = 3.0 * np.sqrt(np.diag(H))
    return H, back[d * d:d * d + d] - pad, back[d * d + d:] + pad


def _candidates(rng, H0, count):
    d = H0.shape[0]
    R = np.linalg.cholesky(H0)
    out = np.empty((count, d, d))
    for i in range(count):
        Q = _rotation(rng, d)
        A = R @ Q @ np.diag(np.exp(rng.uniform(math.log(0.25), math.log(4.0), size=d))) @ Q.T @ R.T
        out[i] = 0.5 * (A + A.T)
    return out


def _opts(case):
    o = {}
    if case["prec"] == "fp64":
        o["precision"] = FP64
    if case.get("rule") == "simple":
        o["binning"] = BIN_SIMPLE
    if case.get("P"):
        o["P_rule"], o["P_fixed"] = P_FIXED, [case["P"]] * case["d"]
    return o


def _inputs(case, seed):
    """Everything that the seed decides."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    d = case["d"]
    if case["kind"] == "many":
        sets = []
        for _ in range(case["sets"]):
            top = case["n"]
            n = max(100, int(round(top * 10.0 ** -rng.uniform(0.0, 2.0))))
            side = case["M0"] if n >= 0.3 * top else case["M0"] // 2 if n >= 0.05 * top else case["M0"] // 4
            X, _ = _sample(rng, gen, n, d, int(rng.integers(2, 5)))
            H, lo, hi = _scale(X)
            sets.append({"X": X, "lo": lo, "hi": hi, "M": [max(16, side)] * d, "H": _candidates(rng, H, case["nH"])})
        return {"sets": sets}
    X, mix = _sample(rng, gen, case["n"], d, 2 + int(rng.integers(0, 3)))
    G, lo, hi = _scale(X)
    H = _candidates(rng, G, case["nH"])
    s = {"X": X, "lo": lo, "hi": hi, "M": _M(case), "G": G, "H": H, "mix": mix}
    if case["kind"] == "analysis":
        s["H"] = G[None].copy()
    if case["kind"] == "autograd":
        s["Ht"] = torch.tensor(H, device="cuda").float()
        s["H"] = s["Ht"].double().cpu().numpy()
        s["w"] = torch.randn(case["nH"], d ** case["r"], generator=gen, device="cuda")
        s["u"] = torch.randn(case["nH"], generator=gen, device="cuda")
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"], s["ctx"], s["o"] = case, _ctx(), _opts(case)
    s["keep"] = np.float32 if case["prec"] == "fp32" else np.float64
    if case["kind"] in ("objective", "kde", "ise", "autograd"):   # the data set that such a program has binned before
        s["ds"] = s["ctx"].bin(s["X"], s["lo"], s["hi"], s["M"], **s["o"])
    if case["kind"] == "kde":
        s["out"] = torch.empty(s["M"], dtype=torch.float64, device="cuda")
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case, ctx, keep = s["case"], s["ctx"], s["keep"]
    kind = case["kind"]
    if kind == "many":
        sets = s["sets"]
        dss = ctx.bin_many([t["X"] for t in sets], [t["lo"] for t in sets], [t["hi"] for t in sets],
                           [t["M"] for t in sets], **s["o"])
        val, grad = ctx.batch_lscv(dss, [t["H"] for t in sets])
        for ds in dss:
            ds.close()
        return {"value": val.astype(keep), "grad": grad.astype(keep)}
    if kind == "objective":
        ds = s["ds"]
        val, grad = ds.lscv(s["H"], grad=True) if case["method"] == "lscv" else ds.scv(s["H"], s["G"], grad=True)
        return {"value": val.astype(keep), "grad": grad.astype(keep)}
    if kind == "kde":   # into the program's own device buffer
        H = np.ascontiguousarray(s["H"][0])
        code = load().kdefft_kde_grid(s["ds"].h, H.ctypes.data, s["out"].data_ptr())
        if code:
            raise RuntimeError(f"kdefft_kde_grid: {code}")
        return {"f": s["out"].float()}
    if kind == "ise":
        w, mu, S = s["mix"]
        return {"ise": s["ds"].ise_mixture(s["H"], w, mu, S).astype(keep)}
    if kind == "autograd":
        H = s["Ht"].detach().requires_grad_()
        psi = ag.psi(s["ds"], H, case["r"])
        psi.backward(s["w"])
        g_psi, H.grad = H.grad, None
        val = ag.lscv(s["ds"], H)
        val.backward(s["u"])
        return {"psi": psi, "psi_grad": g_psi, "value": val, "value_grad": H.grad}
    ds = ctx.bin(s["X"], s["lo"], s["hi"], s["M"], **s["o"])
    if kind == "analysis":
        psi = ds.psi(s["H"], 4)
        val, grad = ds.lscv(s["H"], grad=True)
        out = {"psi": psi.astype(keep), "value": val.astype(keep), "grad": grad.astype(keep)}
    elif kind == "select":
        got = ds.select_H_many([LSCV, SCV], n_starts=case["nstarts"])
        out = {"H": np.stack([g[0] for g in got]).astype(keep), "f": np.array([g[1] for g in got]).astype(keep)}
    elif kind == "psi":
        out = {"psi": ds.psi(s["H"], case["r"]).astype(keep)}
    elif kind == "plugin":
        val, grad = ds.pi(s["H"], s["G"], grad=True)
        out = {"value": val.astype(keep), "grad": grad.astype(keep), "eta02": ds.eta02(s["H"], s["G"]).astype(keep)}
    else:
        whole = case.get("rule") == "simple"
        out = {"counts": ds.counts(DT_I32 if whole else DT_F32 if case["prec"] == "fp32" else DT_F64)}
    ds.close()
    return out


# ------------------------------------------------------------------ work
def _half_box(d, n, M, cover=1.0):
    """Half-box lags of the support of a bandwidth `cover` times the normal
    scale, for a sample of about unit scale on the grid of _scale."""
    h = (4.0 / (d + 2.0)) ** (1.0 / (d + 4.0)) * n ** (-1.0 / (d + 4.0))
    wide = 2.0 * math.sqrt(2.0 * math.log(n)) + 6.0 * h
    pts = 1.0
    for m in M:
        pts *= 2.0 * min(m - 1, math.ceil(TAU * math.sqrt(cover) * h * (m - 1) / wide)) + 1.0
    return 0.5 * pts


def work(case):
    """The sample read and the results written once; per candidate and lag of
    the half box the quadratic form, the exponential and the Hermite values of
    each Gaussian, and a multiply-add per functional; binning: a location and
    2^d weights a point."""
    kind, d, n, M, nH = case["kind"], case["d"], case["n"], _M(case), case["nH"]
    cells = float(np.prod(M))
    keep = 4.0 if case["prec"] == "fp32" else 8.0
    g = d * (d + 1) // 2
    bin_f = n * (6.0 * d + 2.0 ** d * (d + 1))
    bin_b = 8.0 * n * d
    herm = lambda r: math.comb(d + r, d)  # noqa: E731

    def evals(count, nsig, r, outs, cover=2.0):
        return count * _half_box(d, n, M, cover) * (nsig * (2.0 * d * d + 10.0 + 3.0 * herm(r)) + 2.0 * outs)

    if kind == "analysis":
        return {"bytes": bin_b + keep * (d ** 4 + 1 + d * d),
                "flops": bin_f + evals(1, 1, 4, herm(4) - herm(3)) + evals(1, 2, 2, 1 + g)}
    if kind == "select":
        e = 20.0 * case["nstarts"]   # evaluations of a search from each start
        return {"bytes": bin_b + 2 * keep * (d * d + 1), "flops": bin_f + evals(e, 2, 2, 1 + g) + evals(e, 3, 2, 1 + g, 4.0)}
    if kind == "objective":
        f = evals(nH, 2, 2, 1 + g) if case["method"] == "lscv" else evals(nH, 3, 2, 1 + g, 4.0)
        return {"bytes": keep * cells + nH * (8.0 + keep) * d * d + keep * nH, "flops": f}
    if kind == "psi":
        r = case["r"]
        return {"bytes": bin_b + 8.0 * nH * d * d + keep * nH * d ** r,
                "flops": bin_f + evals(nH, 1, r, herm(r) - (herm(r - 1) if r else 0))}
    if kind == "many":
        mean = 0.215 * case["sets"]   # of a log-uniform size over two decades
        return {"bytes": mean * bin_b + case["sets"] * nH * (8.0 + keep) * d * d,
                "flops": mean * bin_f + 0.3 * evals(case["sets"] * nH, 2, 2, 1 + g)}
    if kind == "plugin":
        return {"bytes": bin_b + nH * (8.0 + keep) * d * d + 2 * keep * nH,
                "flops": bin_f + evals(1, 1, 4, herm(4) - herm(3), 1.0) + nH * 4.0 * d ** 4}
    if kind == "kde":
        return {"bytes": (4.0 + 4.0) * cells, "flops": 2.0 * cells * 2.0 * _half_box(d, n, M)}
    if kind == "ise":
        return {"bytes": 4.0 * cells + 8.0 * nH * d * d, "flops": evals(nH, 1, 0, 1) + nH * cells * 3.0 * (2.0 * d * d + 10.0)}
    if kind == "autograd":
        r = case["r"]
        return {"bytes": 4.0 * cells + nH * 4.0 * (2 * d * d + 2 * d ** r),
                "flops": evals(nH, 1, r + 2, herm(r + 2)) + evals(nH, 2, 2, 1 + g)}
    return {"bytes": bin_b + (8.0 if case["prec"] == "fp64" and case.get("rule") != "simple" else 4.0) * cells, "flops": bin_f}


# ------------------------------------------------------------------ 64-bit values
def _counts64(X, lo, hi, M):
    """Linear binning: multilinear weights to the 2^d nodes around a point."""
    n, d = X.shape
    lo, hi = torch.tensor(lo, device="cuda"), torch.tensor(hi, device="cuda")
    top = torch.tensor([m - 1.0 for m in M], dtype=torch.float64, device="cuda")
    t = torch.minimum((X - lo) / ((hi - lo) / top), top)
    l = torch.minimum(torch.floor(t), top - 1.0)
    f = t - l
    l = l.long()
    c = torch.zeros(int(np.prod(M)), dtype=torch.float64, device="cuda")
    for b in itertools.product((0, 1), repeat=d):
        w = torch.ones(n, dtype=torch.float64, device="cuda")
        idx = torch.zeros(n, dtype=torch.int64, device="cuda")
        for k in range(d):
            w = w * (f[:, k] if b[k] else 1.0 - f[:, k])
            idx = idx * M[k] + l[:, k] + b[k]
        c.index_add_(0, idx, w)
    return c.reshape(M)


class _Sums:
    """n^-2 sum_ij c_i c_j k(i - j) over the support box, lags summed first."""

    def __init__(self, X, lo, hi, M):
        self.n, self.d, self.M = X.shape[0], X.shape[1], list(M)
        self.c = _counts64(X, lo, hi, M)
        self.delta = [(float(b) - float(a)) / (m - 1) for a, b, m in zip(lo, hi, M)]
        self.auto = None

    def support(self, B):
        lam = float(np.linalg.eigvalsh(B)[-1])
        return [max(1, int(min(m - 1, math.ceil(TAU * math.sqrt(lam) / dk)))) for m, dk in zip(self.M, self.delta)]

    def box(self, L, widest):
        """Lags x and autocorrelation on |j_k| <= L_k."""
        if self.auto is None:
            A = [min(m - 1, w) for m, w in zip(self.M, widest)]
            P = [m + a for m, a in zip(self.M, A)]
            C = self.c
            dims = tuple(range(self.d))
            C = torch.fft.rfftn(C, s=P, dim=dims)
            self.auto = torch.fft.irfftn(C.real.square() + C.imag.square(), s=P, dim=dims)
        a = self.auto
        for k, Lk in enumerate(L):
            a = torch.cat([a.narrow(k, a.shape[k] - Lk, Lk), a.narrow(k, 0, Lk + 1)], dim=k)
        ax = [self.delta[k] * torch.arange(-Lk, Lk + 1, dtype=torch.float64, device="cuda") for k, Lk in enumerate(L)]
        x = torch.stack([g.reshape(-1) for g in torch.meshgrid(*ax, indexing="ij")])
        return x, a.reshape(-1) / float(self.n) ** 2

    def partials(self, Sigma, x):
        """alpha -> (d^alpha phi_Sigma)(x) for even |alpha|, by the Hermite
        recurrence."""
        Lam = np.linalg.inv(Sigma)
        z = torch.tensor(Lam, device="cuda") @ x
        phi = torch.exp(-0.5 * (x * z).sum(0)) * ((2.0 * math.pi) ** (-0.5 * self.d) / math.sqrt(np.linalg.det(Sigma)))
        memo = {(0,) * self.d: torch.ones_like(phi)}

        def he(al):
            if al not in memo:
                k = next(i for i, v in enumerate(al) if v)
                be = tuple(v - (i == k) for i, v in enumerate(al))
                v = z[k] * he(be)
                for j in range(self.d):
                    if be[j]:
                        v = v - Lam[k, j] * be[j] * he(tuple(w - (i == j) for i, w in enumerate(be)))
                memo[al] = v
            return memo[al]

        return lambda al: phi * he(al)


def _alpha(d, idx):
    a = [0] * d
    for i in idx:
        a[i] += 1
    return tuple(a)


def _k0(S):
    d = S.shape[0]
    return (2.0 * math.pi) ** (-0.5 * d) / math.sqrt(np.linalg.det(S))


def _widest(sums, Bs):
    return [max(v) for v in zip(*[sums.support(B) for B in Bs])]


def _psi64(sums, H, r, widest):
    x, a = sums.box(sums.support(H), widest)
    p = sums.partials(H, x)
    got = {}
    for idx in itertools.product(range(sums.d), repeat=r):
        al = _alpha(sums.d, idx)
        if al not in got:
            got[al] = (p(al) * a).sum()
    return torch.stack([got[_alpha(sums.d, idx)] for idx in itertools.product(range(sums.d), repeat=r)])


def _objective64(sums, H, G, method, widest):
    """Value and tied-entry gradient of LSCV (Eq. 10) or SCV."""
    d, n = sums.d, sums.n
    pairs = [(i, j) for i in range(d) for j in range(i, d)]
    tie = lambda i, j: 1.0 if i == j else 2.0  # noqa: E731
    Hi = np.linalg.inv(H)
    if method == "lscv":
        x, a = sums.box(sums.support(H), widest)
        wide, narrow, const = sums.partials(2.0 * H, x), sums.partials(H, x), None
        k0 = 2.0 * _k0(H) / n
    else:
        x, a = sums.box(sums.support(2.0 * H + 2.0 * G), widest)
        wide, narrow, const = sums.partials(2.0 * H + 2.0 * G, x), sums.partials(H + 2.0 * G, x), sums.partials(2.0 * G, x)
        k0 = (4.0 * math.pi) ** (-0.5 * d) / math.sqrt(np.linalg.det(H)) / n
    z = (0,) * d
    ker = wide(z) - 2.0 * narrow(z)
    if const is not None:
        ker = ker + const(z)
    rows = [(ker * a).sum()]
    for i, j in pairs:
        al = _alpha(d, (i, j))
        rows.append(((wide(al) - narrow(al)) * a).sum())
    r = torch.stack(rows).cpu().numpy()
    g = np.zeros((d, d))
    for v, (i, j) in zip(r[1:], pairs):
        g[i, j] = g[j, i] = tie(i, j) * (v - 0.5 * k0 * Hi[i, j])
    return r[0] + k0, g


def exact(case, seed):
    kind, d = case["kind"], case["d"]
    if kind == "select" or case.get("rule") == "simple":
        return None   # a search's end point has no closed value; whole counts have no error
    s = _inputs(case, seed)
    if kind == "many":
        vals, grads = [], []
        for t in s["sets"]:
            sums = _Sums(t["X"], t["lo"], t["hi"], t["M"])
            wide = _widest(sums, t["H"])
            for H in t["H"]:
                v, g = _objective64(sums, H, None, "lscv", wide)
                vals.append(v)
                grads.append(g)
        return {"value": np.array(vals), "grad": np.array(grads)}
    sums = _Sums(s["X"], s["lo"], s["hi"], s["M"])
    Hs, G = s["H"], s["G"]
    if kind == "bin":
        return {"counts": sums.c.cpu().numpy()}
    if kind == "objective":
        wide = _widest(sums, Hs if case["method"] == "lscv" else [2.0 * H + 2.0 * G for H in Hs])
        got = [_objective64(sums, H, G, case["method"], wide) for H in Hs]
        return {"value": np.array([v for v, _ in got]), "grad": np.array([g for _, g in got])}
    if kind == "analysis":
        v, g = _objective64(sums, Hs[0], None, "lscv", sums.support(Hs[0]))
        return {"psi": _psi64(sums, Hs[0], 4, None).cpu().numpy()[None], "value": np.array([v]), "grad": g[None]}
    if kind == "psi":
        wide = _widest(sums, Hs)
        return {"psi": torch.stack([_psi64(sums, H, case["r"], wide) for H in Hs]).cpu().numpy()}
    if kind == "plugin":
        psi4 = _psi64(sums, G, 4, sums.support(G)).cpu().numpy().reshape(d * d, d * d)
        vals, grads, eta = [], [], []
        for H in Hs:
            q = (H.reshape(-1) @ psi4).reshape(d, d)
            r = (4.0 * math.pi) ** (-0.5 * d) / math.sqrt(np.linalg.det(H)) / sums.n
            eta.append(float((q * H).sum()))
            vals.append(r + 0.25 * eta[-1])
            g = -0.5 * r * np.linalg.inv(H) + 0.5 * q
            grads.append(g * (2.0 - np.eye(d)))
        return {"value": np.array(vals), "grad": np.array(grads), "eta02": np.array(eta)}
    if kind == "kde":
        H = Hs[0]
        L = sums.support(H)
        ax = [sums.delta[k] * torch.arange(-Lk, Lk + 1, dtype=torch.float64, device="cuda") for k, Lk in enumerate(L)]
        x = torch.stack([g.reshape(-1) for g in torch.meshgrid(*ax, indexing="ij")])
        ker = sums.partials(H, x)((0,) * d).reshape([2 * v + 1 for v in L])
        P = [m + 2 * v for m, v in zip(sums.M, L)]
        dims = tuple(range(d))
        f = torch.fft.irfftn(torch.fft.rfftn(sums.c, s=P, dim=dims) * torch.fft.rfftn(ker, s=P, dim=dims), s=P, dim=dims)
        for k, v in enumerate(L):
            f = f.narrow(k, v, sums.M[k])
        return {"f": f / sums.n}
    if kind == "ise":
        w, mu, S = s["mix"]

        def phi(Sg, x):
            z = np.linalg.solve(Sg, x)
            return _k0(Sg) * np.exp(-0.5 * (x * z).sum(0))

        K = len(w)
        ff = sum(w[i] * w[j] * float(phi(S[i] + S[j], (mu[i] - mu[j])[:, None])[0]) for i in range(K) for j in range(K))
        node = [lo + dk * np.arange(m) for lo, dk, m in zip(s["lo"], sums.delta, sums.M)]
        x = np.stack([g.reshape(-1) for g in np.meshgrid(*node, indexing="ij")])
        c = sums.c.cpu().numpy().reshape(-1)
        wide = _widest(sums, [2.0 * H for H in Hs])
        out = []
        for H in Hs:
            cross = sum(w[k] * float(c @ phi(H + S[k], x - mu[k][:, None])) for k in range(K)) / sums.n
            out.append(float(_psi64(sums, 2.0 * H, 0, wide)[0]) - 2.0 * cross + ff)
        return {"ise": np.array(out)}
    # autograd
    r = case["r"]
    wide = _widest(sums, Hs)
    w, u = s["w"].double().cpu().numpy(), s["u"].double().cpu().numpy()
    psi, gpsi, val, gval = [], [], [], []
    for i, H in enumerate(Hs):
        psi.append(_psi64(sums, H, r, wide).cpu().numpy())
        up = _psi64(sums, H, r + 2, wide).cpu().numpy().reshape(d ** r, d, d)
        gpsi.append(0.5 * np.tensordot(w[i], up, axes=1))
        v, g = _objective64(sums, H, None, "lscv", wide)
        val.append(v)
        gval.append(u[i] * g * (0.5 + 0.5 * np.eye(d)))
    return {"psi": np.array(psi), "psi_grad": np.array(gpsi), "value": np.array(val), "value_grad": np.array(gval)}
