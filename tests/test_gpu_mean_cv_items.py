"""All (bandwidth, fold) items of the mean smoother's CV in one launch: one axis and two,
row blocks that do not divide the grid, windows of one bin and of the whole axis, more
bandwidths than one launch holds, empty and single-observation subjects, against the oracle."""
import numpy as np
import pytest

from oracle import cv as ocv

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,nfold,hs", [
    ((5,), 40, 2, [0.15, 0.5, 3.0]),
    ((64,), 90, 5, [0.02, 0.3]),
    ((7, 13), 120, 3, [(0.1, 0.4), (0.9, 0.07), (0.3, 0.3)]),
    ((13, 64), 900, 5, [0.06, 0.33]),
    ((64, 3), 300, 2, [(0.05, 0.5), (0.4, 0.9)]),
    ((6, 6), 100, 2, list(np.linspace(0.2, 1.3, 67))),
])
def test_mean_cv_items_vs_oracle(m, n, nfold, hs):
    from paper_1510_04439_gb300 import binding as B
    ctx = B.Context(0)
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(n + len(hs))
    num = rng.integers(0, 20, size=n)
    num[:2] = (0, 1)
    offs = np.concatenate([[0], np.cumsum(num)]).astype(np.int64)
    t = rng.random((int(offs[-1]), len(m)))
    y = np.sin(3 * t.sum(1)) + 0.3 * rng.standard_normal(len(t))
    fold = (rng.permutation(n) % nfold).astype(np.int32)
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    cv = torch.empty(len(hs), dtype=torch.float64, device=dev)
    ctx.smooth_mean_cv(ctx.sparse(up(offs), up(t), up(y)), m, up(fold), nfold, hs, cv)
    ctx.sync()
    bins = ocv.mean_fold_bins(offs, t, y, m, fold, nfold)
    vec = [h if hasattr(h, "__len__") else [h] * len(m) for h in hs]
    ref = np.array([ocv.mean_cv_score(m, h, *bins) for h in vec])
    got = cv.cpu().numpy()
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    fin = np.isfinite(ref)
    # the same FP64 sums in another order: 1e-9, as the mean CV is held elsewhere
    assert np.all(np.abs(got[fin] - ref[fin]) <= 1e-9 * np.abs(ref[fin]))
