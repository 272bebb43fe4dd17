"""The work that users of this framework have it do, as cases to time and to check.

A case is a dict of plain values with a "kind", one of the framework's entry points
or a short sequence of them:

  fit      the whole plain method in FP64: bins, mean, covariance, full eigenpairs
  gram     covariance bins of gridded data, BF16 products (fpca_bin_cov)
  folds    covariance bins of gridded data split by folds, FP32 (fpca_bin_cov)
  pairs    covariance bins of scattered data split by folds, FP32 (fpca_bin_cov)
  surface  the smoothed covariance surface at one bandwidth (fpca_smooth_cov_project)
  cv       cross-validation of the covariance bandwidths (fpca_smooth_cov_project)
  meancv   cross-validation of the mean bandwidths (fpca_smooth_mean_cv)
  eig      random-projection eigenpairs of a surface (fpca_rproj_eig)
  scores   PACE scores and the reconstruction (fpca_scores_pace, fpca_reconstruct)
  volume   d = 3: factored bins and the smoothed covariance times a block of vectors
  train    one AdamW step of the bandwidth network (fpca_bw_train_step)

Inputs are drawn on the GPU from the observation model of Eq. (2.1)-(2.2) with Fourier
product eigenfunctions.  exact() restates each estimator in FP64 with plain torch.
"""
import math

import torch

from paper_1510_04439_gb300 import binding as B
from paper_1510_04439_gb300 import pipeline

_CTX = None


def _ctx():
    """One library context for the process, as a program that fits many datasets keeps."""
    global _CTX
    if _CTX is None:
        _CTX = B.Context(0)
    return _CTX


def _dev():
    return torch.device("cuda", 0)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # 1-D curves on 64 nodes: the smallest whole fit, where launches and latency count
        {"name": "fit_1d_64", "kind": "fit", "m1": 64, "m2": 0, "n": 100, "h": 0.12, "drop": 0.3,
         "disk": False, "k": 4},
        # n = 50 surfaces on the full 16x16 grid, FP64 throughout, all 256 eigenpairs
        {"name": "fit_2d_16", "kind": "fit", "m1": 16, "m2": 16, "n": 50, "h": 0.15, "drop": 0.0,
         "disk": False, "k": 4},
        # n = 1000 surfaces on 64x64, disk domain, 10% dropped: the dense workload's binning
        {"name": "gram_64", "kind": "gram", "m1": 64, "m2": 64, "n": 1000, "drop": 0.1, "disk": True},
        # the same data split into 5 folds, for cross-validating gridded data
        {"name": "folds_64", "kind": "folds", "m1": 64, "m2": 64, "n": 1000, "drop": 0.1,
         "disk": True, "nfold": 5},
        # n = 20,000 subjects with 5..20 points each on 64x64 bins, 5 folds: longitudinal data
        {"name": "pairs_64", "kind": "pairs", "m1": 64, "m2": 64, "n": 20000, "nfold": 5},
        # the dense workload's surface: 16.8M points, compensated FP32 sums
        {"name": "surface_64", "kind": "surface", "m1": 64, "m2": 64, "n": 1000, "h1": 0.15,
         "h2": 0.15, "comp": True, "drop": 0.1, "disk": True},
        # 16 bandwidths log-spaced over 0.03-0.3 x 5 folds on the longitudinal bins
        {"name": "cv_64", "kind": "cv", "m1": 64, "m2": 64, "n": 20000, "nfold": 5, "nh": 16,
         "lo": 0.03, "hi": 0.3},
        # the same 16 bandwidths for the mean smoother, from the observations
        {"name": "meancv_64", "kind": "meancv", "m1": 64, "m2": 64, "n": 20000, "nfold": 5,
         "nh": 16, "lo": 0.03, "hi": 0.3},
        # rank 8 + 10 oversampling with 2 power iterations on the 4096x4096 surface
        {"name": "eig_64", "kind": "eig", "m1": 64, "m2": 64, "l": 18, "k": 8, "power": 2,
         "disk": True},
        # scores and reconstruction of the dense workload's 1000 surfaces
        {"name": "scores_64", "kind": "scores", "m1": 64, "m2": 64, "n": 1000, "L": 8,
         "drop": 0.1, "disk": True, "sparse": False},
        # n = 2000 volumes on 32x32x32: 1.07e9 covariance points streamed into a 64-column product
        {"name": "volume_32", "kind": "volume", "m1": 32, "m2": 32, "m3": 32, "n": 2000,
         "h": 0.15, "l": 64},
        # one training step of the bandwidth network at its batch of 256
        {"name": "train_256", "kind": "train", "batch": 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng):
    """A grid side of the 2-D workloads: the powers of two that the grids of the
    configurations use, and any other."""
    return rng.choice([32, 64, rng.randint(20, 64), rng.randint(20, 64)])


def draw(rng):
    kind = rng.choice(["fit", "gram", "folds", "pairs", "surface", "surface", "cv", "meancv", "eig",
                       "scores", "volume", "train"])
    if kind == "fit":
        if rng.random() < 0.5:
            m1, m2, h = rng.randint(16, 64), 0, rng.uniform(0.08, 0.2)
        else:
            m1, m2, h = rng.randint(8, 20), rng.randint(8, 20), rng.uniform(0.12, 0.3)
        return {"kind": kind, "m1": m1, "m2": m2, "n": _log(rng, 50, 1000), "h": round(h, 3),
                "drop": rng.choice([0.0, 0.1, 0.3]), "disk": m2 > 0 and rng.random() < 0.3, "k": 4}
    if kind == "train":
        return {"kind": kind, "batch": _log(rng, 1, 1024)}
    if kind == "volume":
        return {"kind": kind, "m1": rng.randint(10, 22), "m2": rng.randint(10, 22),
                "m3": rng.randint(10, 22), "n": _log(rng, 100, 2000),
                "h": round(rng.uniform(0.11, 0.18), 3), "l": rng.choice([8, 18, 33, 64])}
    m1, m2 = _side(rng), _side(rng)
    disk, drop = rng.random() < 0.5, rng.choice([0.0, 0.1, 0.3])
    if kind == "gram":
        # the tensor-core binning takes grids of a multiple of 128 nodes
        m1, m2 = rng.choice([(4 * rng.randint(5, 16), 32), (2 * rng.randint(10, 32), 64),
                             (8 * rng.randint(3, 8), 16 * rng.randint(1, 4))])
        return {"kind": kind, "m1": m1, "m2": m2, "n": _log(rng, 50, 2000), "drop": drop, "disk": disk}
    if kind == "folds":
        return {"kind": kind, "m1": m1, "m2": m2, "n": _log(rng, 50, 1000), "drop": drop,
                "disk": disk, "nfold": rng.choice([2, 5])}
    if kind == "pairs":
        return {"kind": kind, "m1": m1, "m2": m2, "n": _log(rng, 200, 20000),
                "nfold": rng.choice([2, 5])}
    if kind == "surface":
        h1 = round(math.exp(rng.uniform(math.log(0.05), math.log(0.3))), 3)
        h2 = h1 if rng.random() < 0.5 else round(h1 * rng.uniform(0.7, 1.2), 3)
        return {"kind": kind, "m1": m1, "m2": m2, "n": _log(rng, 100, 2000), "h1": h1, "h2": h2,
                "comp": rng.random() < 0.7, "drop": drop, "disk": disk}
    if kind == "cv":
        # three bandwidths are the check of a proposed one, more a search.  Grids on which the
        # library's timed schedules are well apart, so that each run takes the same one (their
        # scores differ in the last bits of FP32)
        m1 = m2 = 64
        if rng.random() < 0.6:
            m1, m2 = rng.randint(20, 48), rng.choice([20, 24, 25, 28, 33, 36, 40, 45, 48])
        return {"kind": kind, "m1": m1, "m2": m2, "n": _log(rng, 2000, 20000),
                "nfold": rng.choice([2, 5]), "nh": rng.choice([1, 3, 3, 9, 16] if m2 == 64 else [1, 3, 3, 4]),
                "lo": round(rng.uniform(0.03, 0.09), 3), "hi": round(rng.uniform(0.15, 0.3), 3)}
    if kind == "meancv":
        return {"kind": kind, "m1": m1, "m2": 0 if rng.random() < 0.3 else m2,
                "n": _log(rng, 200, 20000), "nfold": rng.choice([2, 5]),
                "nh": rng.choice([3, 3, 16]), "lo": round(rng.uniform(0.03, 0.08), 3), "hi": 0.3}
    if kind == "eig":
        k = rng.randint(2, 8)
        return {"kind": kind, "m1": m1, "m2": m2, "l": k + rng.choice([4, 10, 10, 24]), "k": k,
                "power": rng.choice([1, 2, 2]), "disk": disk}
    return {"kind": kind, "m1": m1, "m2": m2, "n": _log(rng, 50, 20000 if m1 * m2 < 600 else 2000),
            "L": rng.choice([2, 4, 8, 8, 13]), "drop": drop, "disk": disk,
            "sparse": rng.random() < 0.4}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _grid(case):
    return tuple(case[a] for a in ("m1", "m2", "m3") if case.get(a, 0) > 0)


def _size(m):
    return int(math.prod(m))


def _gen(seed):
    return torch.Generator(device=_dev()).manual_seed(1510044390 + int(seed))


def _normal(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device=_dev(), dtype=dtype)


def _uniform(g, *shape, dtype=torch.float64):
    return torch.rand(*shape, generator=g, device=_dev(), dtype=dtype)


def _centres(m):
    axes = [(torch.arange(k, device=_dev(), dtype=torch.float64) + 0.5) / k for k in m]
    return torch.stack([a.reshape(-1) for a in torch.meshgrid(*axes, indexing="ij")], 1)


def _phi(pts, count):
    """count orthonormal Fourier products at the points (N x d): N x count."""
    d, out = pts.shape[1], []
    for c in range(count):
        f = torch.ones(pts.shape[0], device=pts.device, dtype=torch.float64)
        for a in range(d):
            x = 2 * math.pi * (1 + (c >> d if a == 0 else 0)) * pts[:, a]
            f = f * math.sqrt(2) * (torch.cos(x) if (c >> a) & 1 else torch.sin(x))
        out.append(f)
    return torch.stack(out, 1)


def _mean(pts):
    if pts.shape[1] == 1:
        return pts[:, 0] + torch.sin(10 * pts[:, 0]) / 10
    if pts.shape[1] == 2:
        return torch.sin(2 * math.pi * pts[:, 0]) * torch.cos(2 * math.pi * pts[:, 1])
    return torch.exp((pts - 0.5).square().sum(1))


def _lam(count):
    return 8.0 * 2.0 ** -torch.arange(count, device=_dev(), dtype=torch.float64)


def _inside(m, disk):
    c = _centres(m)
    return (c - 0.5).square().sum(1) <= 0.25 if disk else torch.ones(c.shape[0], dtype=torch.bool, device=_dev())


def _dense(case, g, mean=True, sigma=0.5, L=6, dtype=torch.float32):
    """Gridded observations y (n x P) and the mask of the observed nodes (uint8)."""
    m, n = _grid(case), case["n"]
    c = _centres(m)
    y = (_normal(g, n, L).double() * _lam(L).sqrt()).to(dtype) @ _phi(c, L).to(dtype).T
    if mean:
        y += _mean(c).to(dtype)
    y += sigma * _normal(g, n, _size(m), dtype=dtype)
    mask = _inside(m, case["disk"]).expand(n, -1)
    if case["drop"] > 0:
        mask = mask & (_uniform(g, n, _size(m), dtype=torch.float32) >= case["drop"])
    return y, mask.to(torch.uint8).contiguous()


def _sparse(case, g, mean=True, L=6):
    """Scattered observations: offs (n + 1), t (N x d), y (N), all on the GPU."""
    m, n = _grid(case), case["n"]
    num = torch.randint(5, 21, (n,), generator=g, device=_dev())
    offs = torch.zeros(n + 1, dtype=torch.int64, device=_dev())
    offs[1:] = num.cumsum(0)
    subj = torch.repeat_interleave(torch.arange(n, device=_dev()), num)
    t = _uniform(g, subj.numel(), len(m))
    y = ((_normal(g, n, L).double() * _lam(L).sqrt())[subj] * _phi(t, L)).sum(1)
    y += 0.5 * _normal(g, subj.numel(), dtype=torch.float64)
    if mean:
        y += _mean(t)
    return offs, t, y


def _folds(case, g):
    return (torch.randperm(case["n"], generator=g, device=_dev()) % case["nfold"]).to(torch.int32)


def _bin(t, m):
    flat = torch.zeros(t.shape[0], dtype=torch.int64, device=t.device)
    for a, k in enumerate(m):
        flat = flat * k + (t[:, a] * k).floor().long().clamp_(0, k - 1)
    return flat


def _symmetric(a):
    return a.triu() + a.triu(1).T


def _pair_weight(num):
    num = num.double()
    return torch.where(num >= 2, 1 / (num * (num - 1)).clamp(min=1), torch.zeros_like(num))


def _bins_dense(y, mask):
    """FP32 covariance bins (counts, W, V) of gridded residuals, as Eq. (2.4) bins them."""
    M = mask.float()
    w = _pair_weight(mask.sum(1)).float()[:, None]
    C, W = M.T @ M, (w * M).T @ M
    V = (w * y * M).T @ (y * M)
    for a in (C, W, V):
        a.fill_diagonal_(0)
    return C.round().to(torch.int32), _symmetric(W), _symmetric(V)


def _bins_sparse(offs, t, r, m, fold, nfold):
    """FP32 fold bins (counts, W, V, Q), each nfold x P x P: the products of each subject's
    binned sums, less the pairs of an observation with itself."""
    P, n = _size(m), offs.numel() - 1
    num = offs[1:] - offs[:-1]
    subj = torch.repeat_interleave(torch.arange(n, device=t.device), num)
    b, w = _bin(t, m), _pair_weight(num)
    out = [torch.empty(nfold, P, P, device=t.device, dtype=torch.int32 if a == 0 else torch.float32)
           for a in range(4)]
    for f in range(nfold):
        who = torch.nonzero(fold == f)[:, 0]
        row = torch.full((n,), -1, dtype=torch.int64, device=t.device)
        row[who] = torch.arange(who.numel(), device=t.device)
        at = torch.nonzero(row[subj] >= 0)[:, 0]
        i, p, x, ww = row[subj[at]], b[at], r[at], w[subj[at]]
        for a in range(4):
            e = (torch.ones_like(x), torch.ones_like(x), x, x * x)[a]
            u = torch.ones_like(x) if a == 0 else ww.sqrt()
            S = torch.zeros(who.numel(), P, device=t.device)
            S.index_put_((i, p), (u * e).float(), accumulate=True)
            G = S.T @ S
            own = torch.zeros(P, device=t.device, dtype=torch.float64)
            own.index_put_((p,), (u * e).square(), accumulate=True)
            G.diagonal().sub_(own.float())
            out[a][f] = G.round().to(torch.int32) if a == 0 else _symmetric(G)
    # bins without a pair hold exact zeros, as the scatter leaves them
    none = out[0] <= 0
    for a in out:
        a.masked_fill_(none, 0)
    return out


def _hs(case):
    nh, d = case["nh"], len(_grid(case))
    if nh == 1:
        return [[case["lo"]] * d]
    r = math.log(case["hi"] / case["lo"]) / (nh - 1)
    return [[case["lo"] * math.exp(r * i)] * d for i in range(nh)]


def _params(g):
    parts = []
    for i, o in _LAYERS:
        parts += [_normal(g, i * o) * math.sqrt(2 / i), 0.01 * _normal(g, o)]
    return torch.cat(parts)


def _surface_like(case, g):
    """A smoothed-covariance-like FP32 surface: sample covariance of n = 1000 smooth curves
    and smoothed noise; NaN where a domain leaves the smoothing window empty."""
    m = _grid(case)
    X = (_normal(g, 1000, 8).double() * _lam(8).sqrt()) @ _phi(_centres(m), 8).T
    e = 0.5 * _normal(g, 1000, *m, dtype=torch.float64)
    for a, k in enumerate(m):
        K = _kernel(k, 0.15)[0]
        e = _along(K / K.sum(1, keepdim=True), e, a + 1)
    X = (X + e.reshape(1000, -1)).float()
    G = _symmetric(X.T @ X / 1000)
    if case["disk"]:
        empty = (_centres(m) - 0.5).square().sum(1).sqrt() > 0.65
        G[empty, :] = float("nan")
        G[:, empty] = float("nan")
    return G


def prepare(case, seed):
    kind, m, g, dev = case["kind"], _grid(case), _gen(seed), _dev()
    P = _size(m) if m else 0
    s = {"case": case, "m": m}
    new = lambda *shape, dtype=torch.float64: torch.empty(*shape, dtype=dtype, device=dev)  # noqa: E731
    if kind == "fit":
        s["y"], s["mask"] = _dense(case, g, L=4, dtype=torch.float64)
        s["bufs"] = pipeline.alloc_dense(torch, dev, P, case["k"], B.F64, B.F64)
    elif kind in ("gram", "folds"):
        y, s["mask"] = _dense(case, g)
        s["y"], s["mu"] = y, _mean(_centres(m)) + 0.05
        F = case.get("nfold", 0)
        shape = (F, P, P) if F else (P, P)
        s["c"] = new(*shape, dtype=torch.int32)
        s["out"] = [new(*shape, dtype=torch.float32) for _ in range(3 if F else 2)]
        s["fold"] = _folds(case, g) if F else None
    elif kind == "pairs":
        s["offs"], s["t"], s["y"] = _sparse(case, g)
        s["fold"], s["mu"] = _folds(case, g), _mean(_centres(m)) + 0.05
        s["c"] = new(case["nfold"], P, P, dtype=torch.int32)
        s["out"] = [new(case["nfold"], P, P, dtype=torch.float32) for _ in range(3)]
    elif kind == "surface":
        s["bins"] = _bins_dense(*_dense(case, g, mean=False))
        s["gamma"], s["status"] = new(P, P, dtype=torch.float32), new(P, P, dtype=torch.uint8)
    elif kind == "cv":
        offs, t, r = _sparse(case, g, mean=False)
        s["bins"] = _bins_sparse(offs, t, r, m, _folds(case, g), case["nfold"])
        s["scores"] = new(case["nh"])
    elif kind == "meancv":
        s["offs"], s["t"], s["y"] = _sparse(case, g)
        s["fold"], s["scores"] = _folds(case, g), new(case["nh"])
    elif kind == "eig":
        s["gamma"], s["domain"] = _surface_like(case, g), _inside(m, case["disk"]).to(torch.int32)
        s["omega"] = _normal(g, P, case["l"])
        s["out"] = [new(case["k"]), new(case["k"], P), new(case["k"])]
    elif kind == "scores":
        L = case["L"]
        if case["sparse"]:
            s["offs"], s["t"], s["y"] = _sparse(case, g, L=L)
        else:
            s["y"], s["mask"] = _dense(case, g, L=L)
        s["mu"], s["phi"], s["lam"] = _mean(_centres(m)), _phi(_centres(m), L).T.contiguous(), _lam(L)
        s["sigma2"] = torch.full((1,), 0.25, dtype=torch.float64, device=dev)
        s["scores"], s["xhat"] = new(case["n"], L), new(case["n"], P, dtype=torch.float32)
    elif kind == "volume":
        s["y"], _ = _dense(dict(case, drop=0.0, disk=False), g, sigma=0.3, L=10)
        s["mu"], s["x"] = _mean(_centres(m)) + 0.05, _normal(g, P, case["l"])
        s["factor"] = new(_ctx().cov_factor_bytes(m, case["n"]), dtype=torch.uint8)
        s["out"] = new(P, case["l"], dtype=torch.float32)
    elif kind == "train":
        b = case["batch"]
        s["feat"], s["target"] = _normal(g, b, 32), 0.5 * _normal(g, b, 6) - 2.2
        s["tmask"] = (_uniform(g, b, 6) < 0.6).to(torch.uint8)
        s["tmask"][0, 0] = 1
        s["params"] = _params(g)
        count = s["params"].numel()
        # the moments of a step in mid-training
        s["m"], s["v"] = 1e-3 * _normal(g, count), 1e-6 * (0.5 + _uniform(g, count, dtype=torch.float32))
        s["step"], s["loss"] = 100, new(1, dtype=torch.float32)
        s["grad"] = new(count, dtype=torch.float32)
    return s


# ---------------------------------------------------------------------------
# one pass through the entry points
# ---------------------------------------------------------------------------

def run(s):
    case, m, ctx = s["case"], s["m"], _ctx()
    kind = case["kind"]
    if kind == "fit":
        h, b = (case["h"],) * len(m), s["bufs"]
        pipeline.run_dense(ctx, m, s["y"], s["mask"], h, h, case["k"], b, bin_prec=B.F64,
                           smooth_prec=B.F64, full=True)
        return {"cnt": b.cnt, "mu": b.mu, "ccnt": b.ccnt, "cv": b.cv, "gamma": b.gamma,
                "status": b.status, "evals": b.evals, "evecs": b.evecs, "fve": b.fve}
    if kind == "gram":
        w, v = s["out"]
        ctx.bin_cov(ctx.dense(s["y"], s["mask"]), m, s["mu"], B.BF16, s["c"], w, v)
        return {"c": s["c"], "w": w, "v": v}
    if kind in ("folds", "pairs"):
        w, v, q = s["out"]
        data = ctx.dense(s["y"], s["mask"]) if kind == "folds" else ctx.sparse(s["offs"], s["t"], s["y"])
        ctx.bin_cov(data, m, s["mu"], B.F32, s["c"], w, v, q=q, fold=s["fold"], nfold=case["nfold"])
        return {"c": s["c"], "w": w, "v": v, "q": q}
    if kind == "surface":
        c, w, v = s["bins"]
        ctx.smooth_cov_project(m, c, w, v, [[case["h1"], case["h2"]]], B.F32C if case["comp"] else B.F32,
                               gamma=s["gamma"], status=s["status"])
        return {"gamma": s["gamma"], "status": s["status"]}
    if kind == "cv":
        c, w, v, q = s["bins"]
        ctx.smooth_cov_project(m, c, w, v, _hs(case), B.F32C, q=q, nfold=case["nfold"], cv=s["scores"])
        return s["scores"]
    if kind == "meancv":
        ctx.smooth_mean_cv(ctx.sparse(s["offs"], s["t"], s["y"]), m, s["fold"], case["nfold"], _hs(case),
                           s["scores"])
        return s["scores"]
    if kind == "eig":
        evals, evecs, fve = s["out"]
        ctx.rproj_eig(m, s["gamma"], case["k"], evals, evecs, fve, domain=s["domain"], omega=s["omega"],
                      power_iters=case["power"])
        return {"evals": evals, "evecs": evecs, "fve": fve}
    if kind == "scores":
        data = ctx.sparse(s["offs"], s["t"], s["y"]) if case["sparse"] else ctx.dense(s["y"], s["mask"])
        ctx.scores_pace(data, m, s["mu"], s["lam"], s["phi"], case["L"], s["sigma2"], s["scores"])
        ctx.reconstruct(m, s["mu"], s["phi"], case["L"], s["scores"], case["n"], s["xhat"])
        return {"scores": s["scores"], "xhat": s["xhat"]}
    if kind == "volume":
        ctx.bin_cov_factor(ctx.dense(s["y"]), m, s["mu"], s["factor"])
        ctx.smooth_cov_apply(m, s["factor"], case["n"], [case["h"]] * 3, s["x"], s["out"])
        return s["out"]
    s["step"] += 1
    ctx.bw_train_step(s["params"], s["m"], s["v"], s["step"], s["feat"], s["target"], s["tmask"],
                      loss=s["loss"], grad=s["grad"])
    return {k: s[k] for k in ("params", "m", "v", "loss", "grad")}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _window(m, h):
    """Mean number of in-grid kernel taps of an axis."""
    return sum(min(m - 1, i + t) - max(0, i - t) + 1 for t in [min(m - 1, math.ceil(h * m) - 1)]
               for i in range(m)) / m


def _smooth_flops(m, h, points):
    """Moment sums of one covariance surface (separable, one axis after another) and its
    local solves, at `points` output pairs."""
    d = len(m)
    if d == 1:
        return points * (2 * 16 * _window(m[0], h[0]) + 40)
    return points * (2 * (6 + 15) * _window(m[0], h[0]) + 2 * (10 + 21) * _window(m[1], h[1]) + 100)


def work(case):
    kind, m = case["kind"], _grid(case)
    P, n = _size(m) if m else 0, case.get("n", 0)
    d, F = len(m), max(1, case.get("nfold", 1))
    half = P * (P + 1) / 2  # the surface is symmetric
    if kind == "fit":
        return {"bytes": 9 * n * P + P * P * (4 + 8 + 8 + 8 + 1),
                "flops": 6 * n * half + _smooth_flops(m, [case["h"]] * d, half) + 4 / 3 * P ** 3}
    if kind in ("gram", "folds"):
        e = 3 if kind == "gram" else 4
        return {"bytes": 5 * n * P + 4 * e * F * P * P, "flops": 2 * e * n * half}
    if kind == "pairs":
        return {"bytes": n * 12.5 * (8 * d + 8) + 16 * F * P * P, "flops": 8 * n * 170}
    if kind == "surface":
        return {"bytes": P * P * (12 + 5), "flops": _smooth_flops(m, (case["h1"], case["h2"]), half)}
    if kind == "cv":
        return {"bytes": 16 * F * P * P, "flops": F * sum(_smooth_flops(m, h, half) for h in _hs(case))}
    if kind == "meancv":
        fit = sum(sum(2 * 3 * (a + 2) * _window(k, h[a]) for a, k in enumerate(m)) + 40 for h in _hs(case))
        return {"bytes": n * 12.5 * (8 * d + 8) + 12 * n, "flops": F * P * fit}
    if kind == "eig":
        l, q = case["l"], case["power"]
        return {"bytes": 4 * P * P + 4 * P * l + 8 * P * case["k"],
                "flops": (q + 2) * (2 * P * P * l + 4 * P * l * l)}
    if kind == "scores":
        L = case["L"]
        obs = n * 12.5 if case["sparse"] else n * P
        return {"bytes": obs * ((8 * d + 8) if case["sparse"] else 5) + n * (8 * L + 4 * P),
                "flops": obs * L * (L + 3) + 2 * n * P * L + n * L ** 3}
    if kind == "volume":
        l, taps = case["l"], [math.ceil(case["h"] * k) - 1 for k in m]
        # pairs whose windows share a node: seven products over the subjects each; the
        # others through the factor, two products of n x P with l columns
        near = math.prod(sum(min(k - 1, i + 2 * t) - max(0, i - 2 * t) + 1 for i in range(k))
                         for k, t in zip(m, taps))
        return {"bytes": 4 * n * P + 8 * P * l, "flops": 14 * n * near / 2 + 8 * n * P * l + 2 * near * l}
    count = sum(i * o + o for i, o in _LAYERS)
    return {"bytes": 4 * count * 7 + 4 * case["batch"] * 44, "flops": 6 * case["batch"] * count + 12 * count}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

_LAYERS = [(32, 256), (256, 256), (256, 256), (256, 6)]


def _kernel(m, h):
    """Epanechnikov weights K(u), K(u) u, K(u) u^2 and the window's indicator, u = (c - x) / h
    with row = output node x, column = bin c: four m x m matrices."""
    i = torch.arange(m, device=_dev(), dtype=torch.float64)
    u = (i[None, :] - i[:, None]) / (h * m)
    k = torch.where(u.abs() < 1, 0.75 * (1 - u * u), torch.zeros_like(u))
    return k, k * u, k * u * u, (u.abs() < 1).double()


def _along(K, x, axis):
    """K applied to one axis of x."""
    if axis == x.dim() - 1:
        return x @ K.T
    a = math.prod(x.shape[:axis])
    return (K @ x.reshape(a, x.shape[axis], -1)).reshape(x.shape)


def _moments(x, K, degree):
    """{exponents: sum K u^e x} over every axis, total degree <= degree."""
    got = {(): x}
    for a in range(len(K)):
        got = {e + (p,): _along(K[a][p], y, a) for e, y in got.items() for p in range(degree - sum(e) + 1)}
    return got


def _fit(cnt, w, v, h):
    """Local linear fit (value, status) at every bin centre of the arrays' grid."""
    m, n = cnt.shape, cnt.dim()
    K = [_kernel(k, h[a]) for a, k in enumerate(m)]
    filled = (cnt > 0).double()
    for a in range(n):
        filled = _along(K[a][3], filled, a)
    S, T = _moments(w, K, 2), _moments(v, K, 1)
    unit = [tuple(int(a == b) for a in range(n)) for b in range(n)]
    e = [(0,) * n] + unit
    A = [[S[tuple(x + y for x, y in zip(e[i], e[j]))] for j in range(i + 1)] for i in range(n + 1)]
    r = [T[x] for x in e]
    low, piv, z = {}, [], []
    bad = filled.round() < n + 1
    for i in range(n + 1):  # LDL' in natural order
        p = A[i][i].clone()
        for k in range(i):
            p -= low[i, k] ** 2 * piv[k]
        bad |= ~(p > 1e-9 * A[i][i])
        piv.append(p)
        x = r[i].clone()
        for k in range(i):
            x -= low[i, k] * z[k]
        z.append(x)
        for j in range(i + 1, n + 1):
            x = A[j][i].clone()
            for k in range(i):
                x -= low[j, k] * low[i, k] * piv[k]
            low[j, i] = x / p
    beta = [None] * (n + 1)
    for i in reversed(range(n + 1)):
        beta[i] = z[i] / piv[i]
        for j in range(i + 1, n + 1):
            beta[i] = beta[i] - low[j, i] * beta[j]
    empty = ~(A[0][0] > 0)
    out = torch.where(bad, r[0] / A[0][0], beta[0])
    out = torch.where(empty, torch.full_like(out, float("nan")), out)
    return out, torch.where(empty, 2, bad.to(torch.int64)).to(torch.uint8)


def _surface(m, c, w, v, h):
    P = _size(m)
    g, st = _fit(c.reshape(m + m), w.double().reshape(m + m), v.double().reshape(m + m), list(h) * 2)
    return g.reshape(P, P), st.reshape(P, P)


def _cv(fit, c, w, v, q):
    """K-fold score of a fit(c, w, v): held-out error over held-out weight."""
    F = c.shape[0]
    ct, wt, vt = c.sum(0), w.double().sum(0), v.double().sum(0)
    err = inn = out = 0.0
    for f in range(F):
        wf, vf = w[f].double(), v[f].double()
        # a bin without pairs in the other folds weighs exactly nothing
        rest = ct - c[f]
        zero = rest <= 0
        g, st = fit(rest, (wt - wf).masked_fill(zero, 0), (vt - vf).masked_fill(zero, 0))
        use = st != 2
        g = torch.where(use, g, torch.zeros_like(g))
        err = err + torch.where(use, q[f].double() - 2 * g * vf + g * g * wf, torch.zeros_like(g)).sum()
        inn, out = inn + wf[use].sum(), out + wf[~use].sum()
    return err / inn if out <= 0.01 * (inn + out) else torch.full_like(err, math.inf)


def _signed(psi):
    big = psi.abs().argmax(0)
    return psi * torch.sign(psi[big, torch.arange(psi.shape[1], device=psi.device)])


def _bins_exact(y, mask, mu):
    M, w = mask.double(), _pair_weight(mask.sum(1))[:, None]
    R = (y.double() - mu) * M
    out = [M.T @ M, (w * M).T @ M, (w * R).T @ R, (w * R * R).T @ (R * R)]
    for a in out:
        a.fill_diagonal_(0)
    out[0] = out[0].round().to(torch.int32)
    return out


def _pairs_exact(s, case):
    """Every ordered pair of two observations of one subject, added into its bin."""
    m, F, P = s["m"], case["nfold"], _size(s["m"])
    num = s["offs"][1:] - s["offs"][:-1]
    n = num.numel()
    subj = torch.repeat_interleave(torch.arange(n, device=_dev()), num)
    b = _bin(s["t"], m)
    r = s["y"] - s["mu"][b]
    w = _pair_weight(num)
    reps = num[subj]  # each observation j with every l of its subject
    j = torch.repeat_interleave(torch.arange(subj.numel(), device=_dev()), reps)
    first = torch.cumsum(reps, 0) - reps
    l = s["offs"][subj[j]] + torch.arange(j.numel(), device=_dev()) - first[j]
    keep = j != l
    j, l = j[keep], l[keep]
    at = (s["fold"][subj[j]].long() * P + b[j]) * P + b[l]
    x, ww = r[j] * r[l], w[subj[j]]
    out = []
    for e in (torch.ones_like(x), ww, ww * x, ww * x * x):
        out.append(torch.zeros(F * P * P, dtype=torch.float64, device=_dev()).index_add_(0, at, e).reshape(F, P, P))
    out[0] = out[0].round().to(torch.int32)
    return out


def _eig_exact(s, case, m):
    P, l, k = _size(m), case["l"], case["k"]
    G, dom = s["gamma"].double(), s["domain"] > 0
    G = torch.nan_to_num(G, nan=0.0) * dom[:, None] * dom[None, :]
    G = (G + G.T) / 2
    Y = G @ s["omega"].double()
    for _ in range(case["power"]):
        Y = G @ torch.linalg.qr(Y)[0]
    Q = torch.linalg.qr(Y)[0]
    B_ = Q.T @ (G @ Q)
    theta, U = torch.linalg.eigh((B_ + B_.T) / 2)
    theta, psi = theta.flip(0)[:k], (Q @ U).flip(1)[:, :k]
    return {"evals": theta / P, "evecs": _signed(psi).T * math.sqrt(P),
            "fve": theta.cumsum(0) / G.diagonal().sum()}


def _fit_exact(s, case, m):
    P, h = _size(m), [case["h"]] * len(m)
    M, y = s["mask"].double(), s["y"]
    num = M.sum(1)
    u = torch.where(num > 0, 1 / num.clamp(min=1), torch.zeros_like(num))
    cnt = M.sum(0)
    mu, _ = _fit(cnt.reshape(m), (u @ M).reshape(m), (u @ (M * y)).reshape(m), h)
    mu = mu.reshape(P)
    C, W, V, _ = _bins_exact(torch.where(s["mask"] > 0, y, torch.zeros_like(y)), s["mask"],
                             torch.nan_to_num(mu, nan=0.0))
    G, st = _surface(m, C, W, V, h)
    dom = cnt > 0
    S = torch.nan_to_num(G, nan=0.0) * dom[:, None] * dom[None, :]
    S = (S + S.T) / 2
    theta, psi = torch.linalg.eigh(S)
    theta, psi = theta.flip(0)[:case["k"]], psi.flip(1)[:, :case["k"]]
    return {"cnt": cnt.to(torch.int32), "mu": mu, "ccnt": C, "cv": V, "gamma": G, "status": st,
            "evals": theta / P, "evecs": _signed(psi).T * math.sqrt(P),
            "fve": theta.cumsum(0) / S.diagonal().sum()}


def _scores_exact(s, case, m):
    phi, lam, L, n = s["phi"].T, s["lam"], case["L"], case["n"]
    if case["sparse"]:
        b = _bin(s["t"], m)
        subj = torch.repeat_interleave(torch.arange(n, device=_dev()), s["offs"][1:] - s["offs"][:-1])
        f = phi[b]
        A = torch.zeros(n, L * L, dtype=torch.float64, device=_dev())
        A.index_add_(0, subj, (f[:, :, None] * f[:, None, :]).reshape(-1, L * L))
        r = torch.zeros(n, L, dtype=torch.float64, device=_dev())
        r.index_add_(0, subj, f * (s["y"] - s["mu"][b])[:, None])
    else:
        M = s["mask"].double()
        A = M @ (phi[:, :, None] * phi[:, None, :]).reshape(-1, L * L)
        r = ((s["y"].double() - s["mu"]) * M) @ phi
    a = torch.linalg.solve(A.reshape(n, L, L) + s["sigma2"] * torch.diag(1 / lam), r)
    return {"scores": a, "xhat": s["mu"] + a @ phi.T}


def _volume_exact(s, case, m):
    P, n = _size(m), case["n"]
    R = (s["y"].double() - s["mu"]) / math.sqrt(n)
    V, W = R.T @ R, torch.ones(P, P, dtype=torch.float64, device=_dev())
    V.fill_diagonal_(0)
    W.fill_diagonal_(0)
    G, _ = _surface(m, W, W, V, [case["h"]] * 3)
    return G @ s["x"].double()


def _train_exact(s, case):
    theta = s["params"].double()
    h, at, used, cache = s["feat"].double(), 0, [], []
    for i, o in _LAYERS:  # weights are used rounded to 16 bits
        W = theta[at:at + i * o].half().double().reshape(i, o)
        b = theta[at + i * o:at + i * o + o]
        at += i * o + o
        z = h @ W + b
        used.append(W)
        cache.append((h, z))
        h = 0.5 * z * (1 + torch.erf(z / math.sqrt(2)))
    M = s["tmask"].double()
    diff = (z - s["target"].double()) * M
    denom = M.sum().clamp(min=1)
    loss, delta, grads = diff.square().sum() / denom, 2 * diff / denom, []
    for i in reversed(range(4)):
        h, z = cache[i]
        grads = [(h.T @ delta).reshape(-1), delta.sum(0)] + grads
        if i:
            z = cache[i - 1][1]
            slope = 0.5 * (1 + torch.erf(z / math.sqrt(2))) + z * torch.exp(-z * z / 2) / math.sqrt(2 * math.pi)
            delta = (delta @ used[i].T) * slope
    grad, t = torch.cat(grads), s["step"] + 1
    m1, v1 = 0.9 * s["m"].double() + 0.1 * grad, 0.999 * s["v"].double() + 0.001 * grad.square()
    up = (m1 / (1 - 0.9 ** t)) / ((v1 / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"params": theta - 1e-3 * (up + 1e-4 * theta), "m": m1, "v": v1, "loss": loss.reshape(1),
            "grad": grad}


def exact(case, seed):
    kind, m = case["kind"], _grid(case)
    if kind == "volume" and _size(m) > 11000:
        return None  # 36 moment arrays of P x P numbers in 64 bits
    s = prepare(case, seed)
    if kind == "fit":
        return _fit_exact(s, case, m)
    if kind == "gram":
        return dict(zip("cwv", _bins_exact(s["y"], s["mask"], s["mu"])))
    if kind == "folds":
        got = [_bins_exact(s["y"][s["fold"] == f], s["mask"][s["fold"] == f], s["mu"])
               for f in range(case["nfold"])]
        return {k: torch.stack([x[a] for x in got]) for a, k in enumerate("cwvq")}
    if kind == "pairs":
        return dict(zip("cwvq", _pairs_exact(s, case)))
    if kind == "surface":
        return dict(zip(("gamma", "status"), _surface(m, *s["bins"], (case["h1"], case["h2"]))))
    if kind == "cv":
        c, w, v, q = s["bins"]
        return torch.stack([_cv(lambda *a: _surface(m, *a, h), c, w, v, q) for h in _hs(case)])
    if kind == "meancv":
        P, F, n = _size(m), case["nfold"], case["n"]
        num = s["offs"][1:] - s["offs"][:-1]
        subj = torch.repeat_interleave(torch.arange(n, device=_dev()), num)
        at = s["fold"][subj].long() * P + _bin(s["t"], m)
        u = (1 / num.double())[subj]
        c, w, v, q = (torch.zeros(F * P, dtype=torch.float64, device=_dev()).index_add_(0, at, x).reshape((F,) + m)
                      for x in (torch.ones_like(u), u, u * s["y"], u * s["y"].square()))
        return torch.stack([_cv(lambda *a: _fit(*a, h), c, w, v, q) for h in _hs(case)])
    if kind == "eig":
        return _eig_exact(s, case, m)
    if kind == "scores":
        return _scores_exact(s, case, m)
    if kind == "volume":
        return _volume_exact(s, case, m)
    return _train_exact(s, case)
