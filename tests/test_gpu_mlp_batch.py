"""The training step's mask count: parts of the mask that are empty, end inside a block's share or
hold every byte value, and a step whose time grows with the batch and not with its square."""
import numpy as np
import pytest

from oracle import mlp as om

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def params(rng):
    return np.concatenate([np.concatenate([rng.standard_normal(i * o) * np.sqrt(2 / i), 0.1 * rng.standard_normal(o)])
                           for i, o in om.LAYERS]).astype(np.float32)


@pytest.mark.parametrize("B,kind", [(1, "none"), (5, "one"), (22, "all"), (23, "bytes"), (457, "tail"), (2000, "bytes")])
def test_loss_denominator(B, kind):
    from paper_1510_04439_gb300 import binding as Bd
    ctx = Bd.Context(0)
    rng = np.random.default_rng(B)
    th = params(rng)
    X, Y = rng.standard_normal((B, 32)).astype(np.float32), rng.standard_normal((B, 6)).astype(np.float32)
    M = {"none": np.zeros((B, 6)), "all": np.ones((B, 6)), "one": np.eye(B, 6) * (np.arange(B)[:, None] == B - 1),
         "tail": np.arange(6 * B).reshape(B, 6) >= 6 * B - 3, "bytes": rng.integers(0, 256, (B, 6))}[kind].astype(np.uint8)
    up = lambda a: torch.from_numpy(a.copy()).to("cuda:0")  # noqa: E731
    p = up(th)
    loss, grad = torch.full((1,), 9.0, device="cuda:0"), torch.full((th.size,), 9.0, device="cuda:0")
    ctx.bw_train_step(p, torch.zeros_like(p), torch.zeros_like(p), 0, up(X), up(Y), up(M), loss=loss, grad=grad)
    ctx.sync()
    want, g = om.loss_and_grad(om.fp16_weights(th), X, Y, (M > 0).astype(np.uint8))
    # FP32 sums of up to 256 terms through four layers, see the rows test
    tol = 4 * 40 * 2.0 ** -24
    assert abs(loss.item() - want) <= 2 * tol * want
    assert np.linalg.norm(grad.cpu().numpy() - g) <= 16 * tol * max(np.linalg.norm(g), 1e-30)


def test_step_time_is_linear():
    from paper_1510_04439_gb300 import binding as Bd
    ctx = Bd.Context(0)
    th = params(np.random.default_rng(0))
    ms = []
    for B in (1 << 17, 1 << 20):
        p = torch.from_numpy(th.copy()).to("cuda:0")
        m, v = torch.zeros_like(p), torch.zeros_like(p)
        X, Y = torch.randn(B, 32, device="cuda:0"), torch.randn(B, 6, device="cuda:0")
        M = (torch.rand(B, 6, device="cuda:0") < 0.6).to(torch.uint8)
        ctx.bw_train_step(p, m, v, 1, X, Y, M)
        ctx.sync()
        ctx.profile(True)
        ctx.bw_train_step(p, m, v, 2, X, Y, M)
        ctx.sync()
        ms.append(ctx.profile_read()["mlp_rows"][0])
        ctx.profile(False)
    # eight times the rows; going through the whole mask in every block took 30 times as long
    assert ms[1] <= 12 * ms[0], ms
