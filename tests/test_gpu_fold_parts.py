"""FP32 fold bins as sums of BF16 part products: folds of 1 to 33 subjects (around the 16 of a
tensor step and the 32 of a stage), grids on and off the 128-node tiles, weights and responses
over many powers of two, and observations whose squares overflow or that are infinite, against
the sums in 64 bits (2e-6 relative and of the largest, the bar of the FP32 binning)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("y32", [False, True])
@pytest.mark.parametrize("m,sizes,odd", [
    ((127,), (1, 15, 17), None),
    ((128,), (16, 33), "range"),
    ((13, 10), (32, 0, 5), None),
    ((130,), (20, 20), "big"),
    ((130,), (20, 20), "inf"),
])
def test_fold_parts(m, sizes, odd, y32):
    from paper_1510_04439_gb300 import binding as B
    P, n, F = int(np.prod(m)), sum(sizes), len(sizes)
    rng = np.random.default_rng(P + n)
    fold = np.repeat(np.arange(F), sizes)
    mu = rng.standard_normal(P)
    y = mu + 2 * rng.standard_normal((n, P))
    mask = rng.random((n, P)) < 0.8
    if odd == "range":
        mask[::3] = rng.random((len(mask[::3]), P)) < 0.05   # weights 300 times the others'
        y *= np.exp2(rng.integers(-20, 21, (1, P)))          # nodes of very different sizes
    if odd == "big":
        y[3, 5], mask[3, 5] = 1e25, True                     # its square is past FP32
    if odd == "inf":
        y[25, 7], mask[25, 7] = np.inf, True
    yv = y.astype(np.float32).astype(np.float64) if y32 else y
    N = mask.sum(1)
    w = np.where(N >= 2, 1.0 / np.maximum(N * (N - 1.0), 1), 0.0)
    r = np.where(mask, yv - mu, 0.0)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")  # noqa: E731
    C = torch.empty(F, P, P, dtype=torch.int32, device="cuda:0")
    W, V, Q = (torch.empty(F, P, P, dtype=torch.float32, device="cuda:0") for _ in range(3))
    ctx = B.Context(0)
    ctx.bin_cov(ctx.dense(dev(y.astype(np.float32) if y32 else y), dev(mask.astype(np.uint8))), m,
                dev(mu), B.F32, C, W, V, q=Q, fold=dev(fold.astype(np.int32)), nfold=F)
    ctx.sync()
    with np.errstate(over="ignore", invalid="ignore"):
        s = np.sqrt(w)[:, None].astype(np.float32)
        x, z = (s * r).astype(np.float32), (s * (r * r).astype(np.float32)).astype(np.float32)
        for f in range(F):
            k = np.nonzero(fold == f)[0]
            M = mask[k].astype(np.float64)
            ref = [M.T @ M, M.T @ (w[k, None] * M), (w[k, None] * r[k]).T @ r[k],
                   (w[k, None] * r[k] ** 2).T @ r[k] ** 2]
            for got, want, parts in ((C, ref[0], None), (W, ref[1], None), (V, ref[2], x), (Q, ref[3], z)):
                got = got[f].cpu().numpy().astype(np.float64)
                np.fill_diagonal(want, 0.0)
                ok = np.ones((P, P), bool)
                if parts is not None:    # where the FP32 sums are no numbers, neither are these
                    t = parts[k].astype(np.float32)
                    bad = ~np.isfinite(t)
                    ok &= ~(bad.any(0)[:, None] | bad.any(0)[None, :])
                    lost = ~ok & ~np.eye(P, dtype=bool)
                    both = (bad.T.astype(int) @ (t != 0).astype(int)) > 0   # an infinity times a number
                    assert not np.isfinite(got[lost & (both | both.T)]).any()
                if odd in ("range",):    # each node by its own size
                    d = np.sqrt(np.maximum(np.abs(want).max(1), 1e-300))
                    assert np.allclose(got / d[:, None] / d, want / d[:, None] / d, rtol=2e-6, atol=2e-5)
                else:
                    top = np.abs(want[ok]).max(initial=1e-300)
                    assert np.allclose(got[ok], want[ok], rtol=2e-6, atol=2e-6 * top), (f, odd)
