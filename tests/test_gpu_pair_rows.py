"""Covariance bins of scattered data summed row by row: rows wider than one CTA's columns,
rows that do not start on 16 bytes, subjects longer than a warp, subjects without pairs,
with and without folds and squared products, against the oracle's pair loop."""
import numpy as np
import pytest

import fpca_synth as fs
from oracle import smoother as sm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("m,n,nmax,nfold,with_q", [
    ((7,), 300, 9, 5, True),         # few rows, many observations in each; P % 4 = 3
    ((8, 8), 60, 70, 3, True),       # subjects longer than a warp
    ((9, 7), 80, 12, 0, False),      # no folds, no squared products
    ((70, 60), 25, 40, 0, True),     # P = 4200: two column blocks in FP32, three in FP64
    ((3, 4, 5), 50, 8, 2, False),    # d = 3
])
def test_pair_rows_vs_oracle(m, n, nmax, nfold, with_q, prec):
    from paper_1510_04439_gb300 import binding as B
    ctx = B.Context(0)
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(sum(m) + n)
    num = rng.integers(0, nmax + 1, size=n)   # some subjects with no or one observation
    num[:2] = (0, 1)
    offs = np.concatenate([[0], np.cumsum(num)]).astype(np.int64)
    t = rng.random((int(offs[-1]), len(m)))
    y = rng.standard_normal(int(offs[-1]))
    mu = np.linspace(-0.4, 0.5, int(np.prod(m)))
    fold = (rng.permutation(n) % max(nfold, 1)).astype(np.int32)
    P, F = int(np.prod(m)), max(nfold, 1)
    dt = torch.float64 if prec == "f64" else torch.float32
    C = torch.full((F, P, P), 7, dtype=torch.int32, device=dev)
    W, V, Q = (torch.full((F, P, P), 3.0, dtype=dt, device=dev) for _ in range(3))
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    ctx.bin_cov(ctx.sparse(up(offs), up(t), up(y)), m, up(mu), B.F64 if prec == "f64" else B.F32,
                C, W, V, q=Q if with_q else None, fold=up(fold) if nfold else None, nfold=nfold)
    ctx.sync()
    r = sm.residuals_sparse(t, y, mu, m)
    c, w, v, q = sm.bin_cov_sparse(offs, t, r, m, fold if nfold else None, nfold)
    assert np.array_equal(C.cpu().numpy(), c)
    # a bin's sum adds at most `most` terms, each rounded to T once and added once
    most = int(c.max()) + 1
    eps = 2.0 ** -53 if prec == "f64" else 2.0 ** -24
    big = np.abs(r).max() ** 2
    for got, ref, scale in ((W, w, 1.0), (V, v, big)) + (((Q, q, big * big),) if with_q else ()):
        bound = 2 * most * eps * scale * w + 1e-300
        assert np.all(np.abs(got.double().cpu().numpy() - ref) <= bound)
    if not with_q:
        assert torch.all(Q == 3.0)
