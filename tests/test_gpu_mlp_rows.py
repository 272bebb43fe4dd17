"""The training step's batch-row kernel and gradient tiles at the edges of their ranges: one
row, rows that do not fill a CTA's share, each number of rows per CTA, batches that do not
fill a staged chunk; gradients only, outputs only; against the FP64 network."""
import numpy as np
import pytest

from oracle import mlp as om

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 2, 3, 63, 65, 304, 305, 608, 613])
def test_step_and_prediction_vs_oracle(B):
    from paper_1510_04439_gb300 import binding as Bd
    ctx = Bd.Context(0)
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(B)
    th = np.concatenate([np.concatenate([rng.standard_normal(i * o) * np.sqrt(2 / i),
                                         0.1 * rng.standard_normal(o)]) for i, o in om.LAYERS])
    th = th.astype(np.float32)
    X = rng.standard_normal((B, 32)).astype(np.float32)
    Y = rng.standard_normal((B, 6)).astype(np.float32)
    M = (rng.random((B, 6)) < 0.6).astype(np.uint8)
    M[0, 0] = 1
    t16 = om.fp16_weights(th)
    out_ref, _ = om.forward(t16, X)
    loss_ref, g_ref = om.loss_and_grad(t16, X, Y, M)
    up = lambda a: torch.from_numpy(a.copy()).to(dev)  # noqa: E731
    out = torch.full((B, 6), 9.0, device=dev)
    ctx.bw_predict(up(th), up(X), out)
    p, m, v = up(th), torch.zeros(th.size, device=dev), torch.zeros(th.size, device=dev)
    loss, grad = torch.empty(1, device=dev), torch.full((th.size,), 9.0, device=dev)
    ctx.bw_train_step(p, m, v, 0, up(X), up(Y), up(M), loss=loss, grad=grad)
    ctx.sync()
    assert np.array_equal(p.cpu().numpy(), th)   # step 0 leaves the parameters
    # FP32 sums of up to 256 terms through four layers: 4 * (256 / 8 + 8) roundings of
    # 2^-24 each, to the norm of each layer's result
    tol = 4 * 40 * 2.0 ** -24
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    assert rel(out.cpu().numpy().astype(float), out_ref) <= tol
    assert abs(loss.item() - loss_ref) <= 2 * tol * loss_ref
    g, at = grad.cpu().numpy().astype(float), 0
    for i, o in om.LAYERS:
        for size in (i * o, o):
            assert rel(g[at:at + size], g_ref[at:at + size]) <= 4 * tol
            at += size
    # one update against the oracle's AdamW on the gradient the GPU formed
    ctx.bw_train_step(p, m, v, 1, up(X), up(Y), up(M), loss=loss, grad=grad)
    ctx.sync()
    th1, m1, v1 = om.adamw_step(th.astype(float), 0 * g, 0 * g, grad.cpu().numpy().astype(float), 1, 1e-3)
    assert np.abs(p.cpu().numpy() - th1).max() <= 1e-6
    assert rel(m.cpu().numpy().astype(float), m1) <= 1e-6
    assert rel(v.cpu().numpy().astype(float), v1) <= 1e-6
