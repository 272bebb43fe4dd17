"""CV sweeps that solve only where held-out pairs are, point by point: the listed fold carries the
score (its squared products, which no fit uses, are a million times the others'), so that one lost
or misplaced point shows; and the sweep that CV runs is chosen by timing CV itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# A term Q - 2 g V + g^2 W is Q to 1e-6 of it, rounded three times; a warp adds 32 lanes of at most
# two, so at most seven additions of it are rounded in FP32: 10 * 2^-24, above and below the
# fraction, with half as much again.
TOL = 2 * 1.5 * 10 * 2.0 ** -24


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def problem(m, per_tile, seed):
    """Bins of three folds: fold 0 with per_tile held-out points in the t-tiles of every fifth s-row,
    two that fill the windows."""
    P, C = m[0] * m[1], m[1]
    rng = np.random.default_rng(seed)
    held = np.zeros((P, P), bool)
    for s in range(0, P, 5):
        for a0 in range(0, m[0], 8):
            tile = np.arange(a0 * C, min(a0 + 8, m[0]) * C)
            tile = tile[tile > s]          # the sweep forms t >= s and mirrors; no own pairs
            if tile.size:
                held[s, rng.choice(tile, min(per_tile, tile.size), replace=False)] = True
    cnt = np.zeros((3, P, P), np.int32)
    cnt[0] = held | held.T
    for f in (1, 2):
        full = np.triu(rng.random((P, P)) < 0.7, 1)
        cnt[f] = full | full.T
    x = rng.standard_normal((3, P, P))
    x = np.triu(x) + np.transpose(np.triu(x, 1), (0, 2, 1))
    W, V, Q = 0.01 * cnt, 0.01 * cnt * x, 0.01 * cnt * x * x
    big = 1e6 * (1 + rng.random((P, P)))
    Q[0] = 0.01 * cnt[0] * (np.triu(big) + np.triu(big, 1).T)
    return cnt, W, V, Q


def score(m, bins, hs, prec, kernel, batch=0):
    from paper_1510_04439_gb300 import binding as B
    ctx = B.Context(0)
    ctx.set_sweep_kernel(kernel)
    ctx.set_cv_batch(batch)
    t = torch.float64 if prec == B.F64 else torch.float32
    out = torch.empty(len(hs), dtype=torch.float64, device="cuda:0")
    c, w, v, q = dev(bins[0]), *(dev(a.astype(np.float32)).to(t) for a in bins[1:])
    ctx.smooth_cov_project(m, c, w, v, hs, prec, q=q, nfold=3, cv=out)
    ctx.sync()
    return out.cpu().numpy()


@pytest.mark.parametrize("nh", [1, 3])
@pytest.mark.parametrize("m,per_tile", [((16, 32), 1), ((16, 32), 47), ((16, 32), 48), ((16, 32), 49),
                                        ((16, 32), 256), ((11, 32), 20), ((8, 64), 2), ((8, 64), 48),
                                        ((8, 64), 200)])
def test_every_listed_point_counts(m, per_tile, nh):
    from paper_1510_04439_gb300 import binding as B
    bins = problem(m, per_tile, per_tile + nh)
    hs = [[(T + 0.5) / m[0], (T + 0.5) / m[1]] for T in (3, 5, 2)[:nh]]
    ref = score(m, bins, hs, B.F64, 0)
    got = score(m, bins, hs, B.F32C, 2)
    assert np.all(np.abs(got - ref) <= TOL * np.abs(ref)), (got, ref)
    # the comparison is sharp: one point (and its mirror) less is far outside the bar
    s, t = np.argwhere(np.triu(bins[0][0]) > 0)[-1]
    for a in bins:
        a[0, s, t] = a[0, t, s] = 0
    less = score(m, bins, hs, B.F64, 0)
    assert np.all(np.abs(less - ref) >= 5 * TOL * np.abs(ref))


def test_cv_is_timed_as_cv():
    from paper_1510_04439_gb300 import binding as B
    m = (16, 32)
    bins = problem(m, 3, 0)
    hs = [[4.5 / 16, 4.5 / 32]]
    ctx = B.Context(0)
    ctx.set_cv_batch(0)
    P = m[0] * m[1]
    c, w, v, q = dev(bins[0]), *(dev(a.astype(np.float32)) for a in bins[1:])
    pool = [c.sum(0).to(torch.int32), w.sum(0), v.sum(0)]
    gamma = torch.empty(P, P, device="cuda:0")
    out = torch.empty(3, 1, dtype=torch.float64, device="cuda:0")
    ctx.smooth_cov_project(m, *pool, hs, B.F32C, gamma=gamma)    # the surface's choice is made
    ctx.sync()
    launched = []
    for k in range(3):
        before = ctx.launches
        ctx.smooth_cov_project(m, c, w, v, hs, B.F32C, q=q, nfold=3, cv=out[k])
        launched.append(ctx.launches - before)
    ctx.sync()
    # the first call times the sweeps on their CV terms, leaving no trace in the score
    assert launched[0] > launched[1] == launched[2]
    got = out.cpu().numpy()[:, 0]
    assert np.all(np.abs(got - got[0]) <= 1e-12 * got[0])
    ref = score(m, bins, hs, B.F64, 0)
    assert np.all(np.abs(got - ref) <= TOL * ref)
