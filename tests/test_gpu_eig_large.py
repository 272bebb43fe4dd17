"""Dense eigenpairs above 256 nodes: the FP64 Jacobi of close eigenvalues runs for the wanted
pairs only.  A smoothed-covariance-like spectrum, whose trailing eigenvalues crowd below FP32's
resolution, leaves it idle; close wanted pairs still get it (or a further refinement step)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solve(A, k):
    from paper_1510_04439_gb300 import binding as B
    n = A.shape[0]
    ctx = B.Context(0)
    out = [torch.empty(s, dtype=torch.float64, device="cuda:0") for s in ((k,), (k, n), (k,))]
    a = torch.from_numpy(np.ascontiguousarray(A)).to("cuda:0")
    ctx.rproj_eig((n,), a, k, *out, full=True)
    ctx.sync()
    ctx.profile(True)
    ctx.rproj_eig((n,), a, k, *out, full=True)
    ctx.sync()
    ms = {name: t for name, (t, _) in ctx.profile_read().items()}
    return out[0].cpu().numpy() * n, out[1].cpu().numpy().T / np.sqrt(n), ms


@pytest.mark.parametrize("n", [257, 324, 400])
def test_smooth_covariance_takes_no_fp64_jacobi(n):
    x = (np.arange(n) + 0.5) / n
    d = x[:, None] - x[None, :]
    A = np.exp(-d * d / 0.02) + 0.1 * np.exp(-np.abs(d) / 0.3)
    lam, psi, ms = solve(A, 4)
    w, V = np.linalg.eigh(A)
    w, V = w[::-1][:4], V[:, ::-1][:, :4]
    assert np.abs(lam - w).max() <= 1e-13 * w[0] * n
    # LAPACK's and ours: some n roundings over the smallest gap each
    assert np.abs(psi * np.sign((psi * V).sum(0)) - V).max() <= 4 * n * 2.0 ** -53 * w[0] / (w[2] - w[3])
    # empty launches against rounds over n x n: a fiftieth here, ten times the rounds when it runs
    assert ms["eig_rotate"] < 0.5 * ms["eig_bj_apply"], ms


@pytest.mark.parametrize("gap", [1e-2, 1e-4, 1e-6, 1e-9])
@pytest.mark.parametrize("n", [257, 324])
def test_close_wanted_pairs(n, gap):
    rng = np.random.default_rng(n)
    Q = np.linalg.qr(rng.standard_normal((n, n)))[0]
    w = 0.5 * 0.9 ** np.arange(n)
    w[:5] = 2 - gap * np.arange(5)
    A = (Q * w) @ Q.T
    A = 0.5 * (A + A.T)
    lam, psi, _ = solve(A, 4)
    assert np.abs(lam - w[:4]).max() <= 1e-12
    assert np.abs(psi.T @ psi - np.eye(4)).max() <= 1e-12
    assert np.abs(A @ psi - psi * lam).max() <= 1e-11
