"""Scratch of the score calls: reconstruction, integration and PACE of scattered data hold the
float-float copies of their functions, not what PACE of gridded data works with; their results
at one block and at many."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def taken(run):
    """Device memory that the context takes over the call (its workspace)."""
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    run()
    torch.cuda.synchronize()
    return free - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("call", ["reconstruct", "integral", "sparse"])
@pytest.mark.parametrize("m,L", [((1, 1), 1), ((3, 85), 2), ((16, 16), 5), ((512, 513), 16)])
def test_scratch_and_values(m, L, call):
    from paper_1510_04439_gb300 import binding as B
    P, n = m[0] * m[1], 4
    g = torch.Generator(device="cuda:0").manual_seed(P)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda:0", dtype=torch.float64)  # noqa: E731
    phi, mu, sc, lam = r(L, P), r(P), r(n, L), 2.0 ** -torch.arange(L, device="cuda:0", dtype=torch.float64)
    ctx = B.Context(0)
    if call == "reconstruct":
        x = torch.empty(n, P, device="cuda:0")
        got = taken(lambda: ctx.reconstruct(m, mu, phi, L, sc, n, x))
        want = mu + sc @ phi
        assert (x.double() - want).abs().max() <= 2 * 2.0 ** -24 * want.abs().max()
    elif call == "integral":
        y, out = r(n, P).float(), torch.empty(n, L, device="cuda:0", dtype=torch.float64)
        data = ctx.dense(y)
        got = taken(lambda: ctx.scores_integral(data, m, mu, phi, L, out))
        want = (y.double() - mu) @ phi.T / P
        assert (out - want).abs().max() <= 1e-12 * (y.double() - mu).abs().max() * phi.abs().max()
    else:
        num = 30
        at = torch.randint(0, P, (n * num,), generator=g, device="cuda:0")
        t = torch.stack([(at // m[1] + 0.5) / m[0], (at % m[1] + 0.5) / m[1]], 1).double()
        y, s2 = r(n * num), torch.full((1,), 0.25, device="cuda:0", dtype=torch.float64)
        offs, out = torch.arange(n + 1, device="cuda:0") * num, torch.empty(n, L, device="cuda:0", dtype=torch.float64)
        data = ctx.sparse(offs, t, y)
        got = taken(lambda: ctx.scores_pace(data, m, mu, lam, phi, L, s2, out))
        f = phi[:, at].T.reshape(n, num, L)
        A = f.transpose(1, 2) @ f + torch.diag(0.25 / lam)
        want = torch.linalg.solve(A, (f * (y - mu[at]).reshape(n, num, 1)).sum(1))
        assert (out - want).abs().max() <= 1e-9 * want.abs().max()
    ctx.sync()
    # two floats a node and function, and a quarter of headroom; allocations in steps of 2 MB
    base = 8 * P * (L + 1)
    assert got <= 1.25 * base + (4 << 20), (got, base)
