"""PACE scores of gridded data on large grids: more nodes than one slab of the table, two batches of
subjects over them, functions that the table does not hold among them, and more node splits than a
launch has blocks in y, against the same systems in 64 bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,L,local", [
    ((257, 130), 37, 3, False),         # 66 splits: tested in a launch of its own
    ((257, 130), 37, 9, True),
    ((513, 513), 130, 3, True),         # a second slab of 17 64s, 112 and 18 subjects
    ((65600, 512), 1, 1, False),        # 65600 splits
])
def test_large_grids(m, n, L, local):
    from paper_1510_04439_gb300 import binding as B
    P = m[0] * m[1]
    g = torch.Generator(device="cuda:0").manual_seed(P % 1000 + L)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda:0", dtype=torch.float64)  # noqa: E731
    phi, mu = r(L, P), r(P)
    if local:
        phi[0] *= 1e-4
        phi[0, 7 * P // 9: 7 * P // 9 + 40] = 20.0
    lam = 2.0 ** -torch.arange(L, device="cuda:0", dtype=torch.float64)
    y = torch.randn(n, P, generator=g, device="cuda:0") + mu.float()
    mask = (torch.rand(n, P, generator=g, device="cuda:0") < 0.7).to(torch.uint8)
    if local:
        mask[::2, 7 * P // 9: 7 * P // 9 + 40] = 0
    out = torch.empty(n, L, device="cuda:0", dtype=torch.float64)
    s2 = torch.full((1,), 0.25, device="cuda:0", dtype=torch.float64)
    ctx = B.Context(0)
    ctx.scores_pace(ctx.dense(y, mask), m, mu, lam, phi, L, s2, out)
    ctx.sync()
    for i in range(n):
        f = phi * mask[i]
        A = f @ f.T + torch.diag(0.25 / lam)
        want = torch.linalg.solve(A, f @ (y[i].double() - mu))
        assert (out[i] - want).abs().max() <= 1e-9 * want.abs().max(), i
