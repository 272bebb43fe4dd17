"""PACE scores of gridded data at the edges of the masks' matrix product: grids that are no
multiple of its 16 and 64 nodes, more subjects than one batch, every count of components
around its column groups, and functions that its fixed-point table does not hold (a spike, a
zero function), against the oracle's N_i x N_i solve."""
import numpy as np
import pytest

from oracle import scores as osc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,L,keep,odd", [
    ((1, 1), 3, 1, 1.0, None),
    ((5, 13), 33, 2, 0.7, None),          # 65 nodes: one past a block of 64
    ((8, 8), 129, 3, 0.5, None),          # one subject past a tile of 128
    ((12, 16), 17, 8, 0.8, "spike"),
    ((16, 16), 40, 8, 0.9, "zero"),
    ((9, 31), 16, 9, 0.9, None),          # two solves per warp, a second pass of columns
    ((20, 20), 31, 13, 0.9, "spike"),
    ((65, 64), 1830, 4, 0.01, None),      # P > 4096: 512 nodes a split, two batches
])
def test_pace_grid_edges(m, n, L, keep, odd):
    from paper_1510_04439_gb300 import binding as B
    P = m[0] * m[1]
    rng = np.random.default_rng(P + 7 * n + L)
    phi = rng.standard_normal((P, L))
    if odd == "spike":
        phi[P // 3, 0] = 300.0            # mean phi^2 of who does not see the node: 4e-6 of the bound
    elif odd == "zero":
        phi[:, L - 1] = 0.0
    lam = 4.0 * 2.0 ** -np.arange(L)
    mu = rng.standard_normal(P)
    y = mu + (rng.standard_normal((n, L)) * np.sqrt(lam)) @ phi.T + 0.5 * rng.standard_normal((n, P))
    mask = (rng.random((n, P)) < keep).astype(np.uint8) * 5   # any nonzero byte is an observation
    if n > 3:
        mask[2] = 0
    ctx = B.Context(0)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")  # noqa: E731
    room = torch.empty(n * P + 1, dtype=torch.uint8, device="cuda:0")
    ref = osc.pace_scores_dense(y, (mask > 0).astype(np.uint8), mu, phi, lam, 0.25)
    for shift in (0, 1):                  # masks that start on and off 16 bytes
        mk = room[shift:shift + n * P].view(n, P)
        mk.copy_(dev(mask))
        out = torch.empty(n, L, dtype=torch.float64, device="cuda:0")
        ctx.scores_pace(B.Context.dense(dev(y), mk), m, dev(mu), dev(lam), dev(phi.T), L,
                        dev(np.array([0.25])), out)
        ctx.sync()
        assert np.max(np.abs(out.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref)), (m, shift)
