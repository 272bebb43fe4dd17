"""CV sweeps that solve only where held-out pairs are: tiles of 8 x 32 points with no such
point, one, 48 (the longest list), 49 and all of them, against the FP64 smoother on the same
bins (1e-4, the bar of FP32 CV scores); and the FP64 covariance bins of gridded data around
their 8 x 8 tiles and runs of 32 and 256 subjects, against the sums in 64 bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


@pytest.mark.parametrize("kernel", [1, 2])
@pytest.mark.parametrize("nh", [1, 4])
@pytest.mark.parametrize("per_tile", [0, 1, 48, 49])
def test_cv_lists(per_tile, nh, kernel):
    from paper_1510_04439_gb300 import binding as B
    m = (16, 32)
    P = 512
    rng = np.random.default_rng(per_tile)
    held = np.zeros((P, P), bool)
    for s in range(0, P, 5):                 # the tiles of every fifth row
        for t1 in (0, 8):
            at = rng.choice(256, per_tile, replace=False)
            held[s, t1 * 32 + at] = True
    held = np.triu(held) | np.triu(held, 1).T
    C = np.zeros((3, P, P), np.int32)        # the fold above, and two that fill the windows
    C[0] = held
    for f in (1, 2):
        full = np.triu(rng.random((P, P)) < 0.7)
        C[f] = full | np.triu(full, 1).T
    for f in range(3):
        np.fill_diagonal(C[f], 0)
    x = rng.standard_normal((3, P, P))
    x = np.triu(x) + np.transpose(np.triu(x, 1), (0, 2, 1))
    W, V, Q = 0.01 * C, 0.01 * C * x, 0.01 * C * x * x
    hs = [[2 * a, a] for a in (0.14, 0.17, 0.2, 0.23)[:nh]]   # 4..7 taps on both axes
    got = {}
    for prec, t in ((B.F32C, torch.float32), (B.F64, torch.float64)):
        ctx = B.Context(0)
        ctx.set_sweep_kernel(kernel)
        ctx.set_cv_batch(0)
        out = torch.empty(nh, dtype=torch.float64, device="cuda:0")
        bins = [dev(a.astype(np.float32)).to(t) for a in (W, V, Q)]
        ctx.smooth_cov_project(m, dev(C), bins[0], bins[1], hs, prec, q=bins[2], nfold=3, cv=out)
        ctx.sync()
        got[prec] = out.cpu().numpy()
    assert np.allclose(got[B.F32C], got[B.F64], rtol=1e-4, atol=0, equal_nan=True)


@pytest.mark.parametrize("P,n", [(1, 3), (7, 31), (8, 32), (9, 33), (65, 257)])
def test_cov_dense_f64_tiles(P, n):
    from paper_1510_04439_gb300 import binding as B
    rng = np.random.default_rng(P + n)
    y, mu = rng.standard_normal((n, P)), rng.standard_normal(P)
    mask = (rng.random((n, P)) < 0.7).astype(np.uint8)
    mask[0] = 0
    C = torch.empty(P, P, dtype=torch.int32, device="cuda:0")
    W, V = (torch.empty(P, P, dtype=torch.float64, device="cuda:0") for _ in range(2))
    ctx = B.Context(0)
    ctx.bin_cov(ctx.dense(dev(y), dev(mask)), (P,), dev(mu), B.F64, C, W, V)
    ctx.sync()
    M, N = mask.astype(np.float64), mask.sum(1).astype(np.float64)
    w = np.where(N >= 2, 1.0 / np.maximum(N * (N - 1), 1), 0.0)[:, None]
    R = np.where(mask > 0, y - mu, 0.0)
    off = ~np.eye(P, dtype=bool)
    assert np.array_equal(C.cpu().numpy(), np.where(off, M.T @ M, 0).astype(np.int32))
    for got, want in ((W, M.T @ (w * M)), (V, (w * R).T @ R)):
        want = np.where(off, want, 0.0)
        # n roundings of 2^-53 of at most the sum of magnitudes
        assert np.abs(got.cpu().numpy() - want).max() <= 4 * n * 2.0 ** -53 * np.abs(R).max() ** 2 * n
