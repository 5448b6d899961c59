"""The whole-network surrogate kernels at the edges of their tiles: widths and
input counts that are not multiples of the tensor core's or the vector copies'
sizes, batches just past a 128-row tile, and widths beyond the kernels' (which
the layer-by-layer path takes).  The gradient and the prediction against the
FP64 network with the operands' BF16 rounding left out, by the other surrogate
tests' bars (2e-2 forward, 3e-2 gradient), and tcgen05 against mma.sync."""
import numpy as np
import pytest

from oracle import mlp
from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,H,n", [(8, 16, 1), (45, 64, 127), (32, 256, 129), (17, 48, 300), (192, 256, 1000),
                                   (256, 256, 130), (32, 272, 140), (300, 64, 128)])
def test_gradient_and_prediction(K, H, n):
    from paper_1905_12795_gb300 import binding as B
    ctx = B.Context([B.make_grid(41, 41, 10.0, 10.0, 5, 4, 0.2, 10.0, 1500.0, 3000.0)],
                    synth.receiver_line(41, 10.0, 20.0), B.EmpsoPso(1024, K, 1.2, 2.9, 0.5, 0.3, 0.25, 10, 1, 7),
                    1200.0, 3200.0)
    ctx.surrogate_init(hidden=H, capacity=64, lr=1e-3, seed=5)
    npar = ctx.surrogate_n_params()
    w = torch.zeros(npar, device="cuda")
    ctx.surrogate_get(w)
    rng = np.random.default_rng(K + H + n)
    bias = torch.tensor(rng.normal(size=npar).astype(np.float32) * 0.05, device="cuda")
    ctx.surrogate_set(w + bias)
    prm = mlp.unflatten((w + bias).cpu().numpy().astype(np.float64), K, H)
    x = rng.uniform(1200.0, 3200.0, size=(n, K)).astype(np.float32)
    t = rng.normal(size=n).astype(np.float32)
    xn = mlp.to_bf16(2.0 * (x.astype(np.float64) - 1200.0) / 2000.0 - 1.0)
    y = mlp.forward(prm, xn)[0]
    out = {}
    for backend in (1, 0):
        ctx.surrogate_set_backend(backend)
        g, loss = torch.zeros(npar, device="cuda"), torch.zeros(1, device="cuda")
        p = torch.zeros(n, device="cuda")
        ctx.surrogate_predict(torch.tensor(x, device="cuda"), p)
        ctx.surrogate_grad(torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda"), g, loss)
        out[backend] = p.cpu().numpy(), g.cpu().numpy(), loss.item()
    assert ctx.device_error() == 0
    ctx.close()
    p, g, loss = out[1]
    assert np.allclose(p, y, rtol=2e-2, atol=2e-2 * max(1.0, np.abs(y).max()))
    assert loss == pytest.approx(0.5 * np.mean((p - t) ** 2), rel=1e-4)
    # the same BF16 products in another order: FP32 rounding of sums of up to n terms
    for a, b in zip(out[1][:2], out[0][:2]):
        assert np.linalg.norm(a - b) <= 2e-4 * np.linalg.norm(b)
