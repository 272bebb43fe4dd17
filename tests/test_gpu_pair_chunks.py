"""Covariance bins of scattered data whose rows hold many observations: chunks of a row added to
the cleared row, at and around the chunk's length, on one bin, few bins and one crowded bin of
many, against the oracle's pair loop; and a crowded bin does not hold up the call."""
import numpy as np
import pytest

from oracle import smoother as sm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def bins(ctx, offs, t, y, m, fold, nfold, prec, with_q=True):
    from paper_1510_04439_gb300 import binding as B
    P, F = int(np.prod(m)), max(nfold, 1)
    dt = torch.float64 if prec == B.F64 else torch.float32
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")  # noqa: E731
    C = torch.full((F, P, P), 7, dtype=torch.int32, device="cuda:0")
    W, V, Q = (torch.full((F, P, P), 3.0, dtype=dt, device="cuda:0") for _ in range(3))
    args = (ctx.sparse(up(offs), up(t), up(y)), m, up(np.zeros(P)), prec, C, W, V)
    kw = dict(q=Q if with_q else None, fold=up(fold) if nfold else None, nfold=nfold)
    ctx.bin_cov(*args, **kw)
    ctx.sync()
    return (C, W, V, Q), lambda: ctx.bin_cov(*args, **kw)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("m,crowd,nfold,with_q", [
    ((1,), 256, 0, True),          # one row of one chunk
    ((1,), 257, 0, True),          # one observation past it
    ((3,), 512, 2, True),
    ((3,), 513, 2, False),
    ((16,), 1500, 0, True),
    ((9, 7), 700, 3, True),        # P % 4 = 3
    ((70, 60), 600, 0, True),      # more than one block of columns
])
def test_long_rows_vs_oracle(m, crowd, nfold, with_q, prec):
    from paper_1510_04439_gb300 import binding as B
    rng = np.random.default_rng(crowd + sum(m))
    num = rng.integers(2, 40, size=max(8, crowd // 20))
    if m == (1,):                  # the row's exact length
        num = np.full(crowd // 8, 8)
        num[0] += crowd % 8
    offs = np.concatenate([[0], np.cumsum(num)]).astype(np.int64)
    N, n = int(offs[-1]), num.size
    t = rng.random((N, len(m)))
    at = rng.permutation(N)[:min(crowd, N)]
    t[at] = 0.5                    # the crowded bin
    y = rng.standard_normal(N)
    fold = (rng.permutation(n) % max(nfold, 1)).astype(np.int32)
    got, _ = bins(B.Context(0), offs, t, y, m, fold, nfold, B.F64 if prec == "f64" else B.F32, with_q)
    c, w, v, q = sm.bin_cov_sparse(offs, t, y, m, fold if nfold else None, nfold)
    assert np.array_equal(got[0].cpu().numpy(), c)
    # a bin's sum adds at most `most` terms, each rounded to T once and added once
    most = int(c.max()) + 1
    eps = 2.0 ** -53 if prec == "f64" else 2.0 ** -24
    big = np.abs(y).max() ** 2
    for a, ref, scale in ((got[1], w, 1.0), (got[2], v, big)) + (((got[3], q, big * big),) if with_q else ()):
        assert np.all(np.abs(a.double().cpu().numpy() - ref) <= 2 * most * eps * scale * w + 1e-300)
    if not with_q:
        assert torch.all(got[3] == 3.0)


def test_crowded_bin_does_not_hold_up_the_call():
    from paper_1510_04439_gb300 import binding as B
    rng = np.random.default_rng(0)
    n = 20000
    num = rng.integers(5, 21, size=n)
    offs = np.concatenate([[0], np.cumsum(num)]).astype(np.int64)
    N = int(offs[-1])
    y, t = rng.standard_normal(N), rng.random((N, 2))
    ms = []
    for crowded in (False, True):
        if crowded:
            t[rng.random(N) < 0.5] = 0.4
        ctx = B.Context(0)
        _, again = bins(ctx, offs, t, y, (48, 48), None, 0, B.F32)
        ctx.profile(True)
        for _ in range(3):
            again()
        ctx.sync()
        ms.append(ctx.profile_read()["cov_rows"][0])
    # the same number of pairs; one CTA per row took twenty times as long
    assert ms[1] <= 5 * ms[0], ms
