"""Offsets of scattered data that decrease: the subject is reported and skipped, neighbours
that then overlap share no observation, every other fold is right, and the context goes on
working."""
import numpy as np
import pytest

from oracle import smoother as sm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def claims(offs, N):
    """How often each observation is claimed by a subject of at least two in 0..N."""
    got = np.zeros(N, int)
    for lo, hi in zip(offs[:-1], offs[1:]):
        if 0 <= lo <= hi <= N and hi - lo >= 2:
            got[lo:hi] += 1
    return got


@pytest.mark.parametrize("m", [(16,), (9, 7)])
@pytest.mark.parametrize("bad", [[0, 10, 5, 12], [0, 20, 10, 30], [0, 40, 0, 40, 1, 40], [0, 3, 1, 9], [0, 60, 6]])
def test_overlapping_offsets(bad, m):
    from paper_1510_04439_gb300 import binding as B
    ctx = B.Context(0)
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(len(bad) + sum(m))
    # good subjects of fold 1 in front, the malformed run (fold 0) after them
    num = rng.integers(0, 15, size=200)
    good = np.concatenate([[0], np.cumsum(num)]).astype(np.int64)
    at = int(good[-1])
    offs = np.concatenate([good[:-1], at + np.array(bad)]).astype(np.int64)
    n = offs.size - 1
    fold = np.where(np.arange(n) < 200, 1, 0).astype(np.int32)
    offs = np.concatenate([offs, [max(at + max(bad), offs[-1])]])   # offs[n] covers them all
    fold = np.concatenate([fold, [0]]).astype(np.int32)
    N = int(offs[-1])
    assert not np.all(np.diff(offs) >= 0)
    if bad[:3] in ([0, 10, 5], [0, 20, 10]):
        assert claims(offs, N).max() == 2
    t, y = rng.random((N, len(m))), rng.standard_normal(N)
    mu = np.zeros(int(np.prod(m)))
    P = mu.size
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    C = torch.empty(2, P, P, dtype=torch.int32, device=dev)
    W, V, Q = (torch.empty(2, P, P, dtype=torch.float64, device=dev) for _ in range(3))

    def run(o, f):
        ctx.bin_cov(ctx.sparse(up(o), up(t), up(y)), m, up(mu), B.F64, C, W, V, q=Q, fold=up(f), nfold=2)

    run(offs, fold)
    with pytest.raises(B.FpcaError):
        ctx.sync()
    want = sm.bin_cov_sparse(good, t, y, m, np.ones(200, np.int32), 2)
    assert np.array_equal(C[1].cpu().numpy(), want[0][1])
    for got, ref in ((W, want[1]), (V, want[2]), (Q, want[3])):
        assert np.allclose(got[1].cpu().numpy(), ref[1], rtol=1e-12, atol=1e-12)
    # each claimed observation pairs with its subject's others once at most
    most = sum((hi - lo) * (hi - lo - 1) for lo, hi in zip(offs[200:-1], offs[201:]) if 0 <= lo <= hi <= N)
    assert 0 <= int(C[0].sum()) <= most
    run(good, np.ones(200, np.int32))
    ctx.sync()
    assert np.array_equal(C[1].cpu().numpy(), want[0][1])
    assert int(C[0].abs().sum()) == 0
