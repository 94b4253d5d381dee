"""The cost model's forward pass, loss and gradients at the batch sizes where
the launch changes (one sample, a partly filled CTA, one CTA, one cluster at 8,
16 and 32 samples a CTA, several clusters), against FP64 autograd.  The sums
have at most 64 FP32 terms per layer and at most 32 per partial gradient, so
1e-5 of the largest value is about fifty roundings of the largest term."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_16940_gb300 as q
    return q


@pytest.mark.parametrize("n", [1, 7, 8, 9, 64, 65, 128, 129, 256, 257, 777, 2500])
def test_loss_grad_and_forward(q, n):
    rng = np.random.default_rng(n)
    P = q.qsa_costmodel_init(3) + rng.normal(0, 0.02, q.MLP_PARAMS).astype(np.float32)
    X = rng.random((n, 37)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    dP, dX, dt = (torch.from_numpy(v).cuda() for v in (P, X, t))
    G = torch.full((q.MLP_PARAMS,), 7.0, device="cuda")
    L, y = torch.full((1,), 7.0, device="cuda"), torch.empty(n, device="cuda")
    ws = torch.empty(q.qsa_mlp_workspace_bytes(n) // 4, device="cuda")
    q.qsa_mlp_loss_grad(dP.data_ptr(), dX.data_ptr(), dt.data_ptr(), n, G.data_ptr(), L.data_ptr(), ws.data_ptr())
    G0 = G.clone()
    q.qsa_mlp_loss_grad(dP.data_ptr(), dX.data_ptr(), dt.data_ptr(), n, G.data_ptr(), 0, ws.data_ptr())
    assert torch.equal(G, G0)   # deterministic, with and without the loss
    q.qsa_mlp_forward(dP.data_ptr(), dX.data_ptr(), n, y.data_ptr(), ws.data_ptr())
    p = dP.double().requires_grad_()
    w1, b1, w2, b2, w3, b3 = torch.split(p, [64 * 37, 64, 64 * 64, 64, 64, 1])
    a = torch.relu(dX.double() @ w1.view(64, 37).T + b1)
    out = torch.relu(a @ w2.view(64, 64).T + b2) @ w3 + b3
    loss = ((out - dt.double()) ** 2).mean()
    loss.backward()
    assert (y.double() - out).abs().max() <= 1e-5 * out.abs().max()
    assert abs(L.item() - loss.item()) <= 1e-5 * loss.item()
    assert (G.double() - p.grad).abs().max() <= 1e-5 * p.grad.abs().max()
