"""Dense eigenpairs on grids of up to 256 nodes: paddings to 32, one block pair and eight,
spectra with close and with equal eigenvalues, null spaces, every eigenpair at once, and
the large-grid path, against the oracle's dense solver."""
import numpy as np
import pytest

from oracle import eigen as oe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def spectrum(kind, n, rng):
    if kind == "decay":
        return 8.0 * 0.7 ** np.arange(n)
    if kind == "flat":          # neighbours 2e-3 / n apart
        return 1.0 + 2e-3 * np.arange(n)[::-1] / n
    if kind == "pairs":         # pairs 1e-6 apart
        return np.repeat(np.arange(n, 0, -1.0), 2)[:n] + 1e-6 * (np.arange(n) % 2 == 0)
    if kind == "lowrank":
        return np.where(np.arange(n) < 3, 3.0 - np.arange(n), 0.0)
    return np.sort(rng.standard_normal(n))[::-1]   # both signs


@pytest.mark.parametrize("kind", ["decay", "flat", "pairs", "lowrank", "signs"])
@pytest.mark.parametrize("m,k", [((1,), 1), ((5,), 5), ((32,), 4), ((33,), 7), ((8, 8), 4),
                                 ((16, 16), 4), ((16, 16), 256), ((17, 16), 5)])
def test_dense_eigenpairs_vs_oracle(m, k, kind):
    from paper_1510_04439_gb300 import binding as B
    ctx = B.Context(0)
    dev = torch.device("cuda", 0)
    n = int(np.prod(m))
    rng = np.random.default_rng(n + k)
    Q = np.linalg.qr(rng.standard_normal((n, n)))[0]
    w = spectrum(kind, n, rng)
    A = (Q * w) @ Q.T
    A = 0.5 * (A + A.T)
    ev = torch.empty(k, dtype=torch.float64, device=dev)
    vec = torch.empty(k, n, dtype=torch.float64, device=dev)
    fve = torch.empty(k, dtype=torch.float64, device=dev)
    ctx.rproj_eig(m, torch.from_numpy(A).to(dev), k, ev, vec, fve, full=True)
    ctx.sync()
    lam, phi, _ = oe.eig_full(A, m, np.ones(n, bool), k)
    big = np.abs(w).max() / n
    got = ev.cpu().numpy()
    assert np.all(np.abs(got - lam) <= 1e-10 * big)
    psi = vec.cpu().numpy().T / np.sqrt(n)
    # residuals and orthonormality hold for any basis of an eigenspace
    assert np.abs(psi.T @ psi - np.eye(k)).max() <= 1e-9
    assert np.abs(A @ psi - psi * (got * n)).max() <= 1e-8 * np.abs(w).max()
