"""The bench counts the points that CV solves, not those of the whole surfaces."""
import pytest

torch = pytest.importorskip("torch")


def test_points_with_held_out_pairs():
    import bench
    w = torch.zeros(3, 6, 6)
    v, q = w.clone(), w.clone()
    w[0, 1, 4] = w[0, 4, 1] = 0.5           # a pair and its mirror
    v[1, 2, 2] = -1.0                       # on the diagonal, weight lost to rounding
    q[2, 5, 0] = q[2, 0, 5] = 1e-30
    w[2, 5, 0] = w[2, 0, 5] = 0.1
    assert bench.held_out_points(torch, w, v, q) == (5, 3)
    assert bench.held_out_points(torch, torch.ones(2, 4, 4), torch.zeros(2, 4, 4), torch.zeros(2, 4, 4)) == (32, 20)
