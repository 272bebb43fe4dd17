"""Dense eigenpairs of surfaces on any scale: what FP32 cannot square (2^70), cannot hold (2^140,
2^600) or takes for nothing (2^-90, 2^-600) has the same eigenvectors, and eigenvalues that are
exactly as much larger; surfaces that are not finite have NaN eigenpairs and leave the context
working.  On both sides of the 256 nodes where the solver changes."""
import numpy as np
import pytest

from oracle import eigen as oe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solve(A, m, k):
    from paper_1510_04439_gb300 import binding as B
    ctx = B.Context(0)
    out = [torch.full(s, 7.0, dtype=torch.float64, device="cuda:0") for s in ((k,), (k, A.shape[0]), (k,))]
    ctx.rproj_eig(m, torch.from_numpy(np.ascontiguousarray(A)).to("cuda:0"), k, *out, full=True)
    ctx.sync()
    return [a.cpu().numpy() for a in out]


def matrix(n, kind):
    rng = np.random.default_rng(n)
    Q = np.linalg.qr(rng.standard_normal((n, n)))[0]
    w = 8.0 * 0.7 ** np.arange(n) if kind == "decay" else np.sort(rng.standard_normal(n))[::-1]
    A = (Q * w) @ Q.T
    return 0.5 * (A + A.T), np.abs(w).max()


@pytest.mark.parametrize("kind", ["decay", "signs"])
@pytest.mark.parametrize("m,k", [((5,), 3), ((8, 8), 4), ((16, 16), 4), ((17, 17), 4)])
@pytest.mark.parametrize("e", [70, 140, 600, -90, -600])
def test_scaled_surface(m, k, kind, e):
    n = int(np.prod(m))
    A, big = matrix(n, kind)
    lam, phi, _ = oe.eig_full(A, m, np.ones(n, bool), k)
    ev, vec, fve = solve(np.ldexp(A, e), m, k)
    # the bars of the unscaled surfaces
    assert np.all(np.abs(np.ldexp(ev, -e) - lam) <= 1e-10 * big / n)
    psi = vec.T / np.sqrt(n)
    assert np.abs(psi.T @ psi - np.eye(k)).max() <= 1e-9
    assert np.abs(A @ psi - psi * (np.ldexp(ev, -e) * n)).max() <= 1e-8 * big
    assert np.allclose(fve, np.cumsum(lam) * n / np.trace(A), rtol=1e-9, atol=0)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, 1e308])
@pytest.mark.parametrize("m,k", [((5,), 5), ((8, 8), 4), ((16, 16), 256), ((17, 17), 4)])
def test_surface_not_finite(m, k, bad):
    n = int(np.prod(m))
    A, big = matrix(n, "decay")
    if np.isfinite(bad):   # its symmetrised entry is not
        A[1, 2] = A[2, 1] = 1.7e308
    else:
        A[1, 2] = A[2, 1] = bad
        A[3, 3] = np.inf
    ev, vec, fve = solve(A, m, k)
    assert np.isnan(ev).all() and np.isnan(vec).all() and np.isnan(fve).all()
    A, big = matrix(n, "decay")
    ev, _, _ = solve(A, m, k)
    lam = oe.eig_full(A, m, np.ones(n, bool), k)[0]
    assert np.all(np.abs(ev - lam) <= 1e-10 * big / n)
