"""The replay targets' mean and standard deviation, summed by a cluster of CTAs:
buffers so short that most of its CTAs have no row and reach their store to the
first one's shared memory at once, at the edges of a CTA's and the cluster's
threads, and past the buffer's capacity."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cap", [(1, 64), (2, 64), (511, 4096), (513, 4096), (4096, 4096), (4097, 8192), (300, 256)])
def test_standardisation_of_short_and_full_buffers(n, cap):
    from paper_1905_12795_gb300 import binding as B
    K = 12
    grid = B.make_grid(41, 41, 10.0, 10.0, 5, 4, 0.2, 10.0, 1500.0, 3000.0, kx=4, kz=3)
    ctx = B.Context([grid], [[0.0, 0.0]], B.EmpsoPso(16, K, 1.2, 2.9, 0.5, 0.3, 0.25, 1, 1, 7), 1500.0, 3000.0)
    ctx.surrogate_init(64, cap, 1e-3, 3)
    rng = np.random.default_rng(n)
    x = rng.uniform(1500.0, 3000.0, (n, K)).astype(np.float32)
    f = np.exp(rng.normal(1.0, 2.0, n))
    p0, p1 = (torch.zeros(16, device="cuda") for _ in range(2))
    q = torch.tensor(rng.uniform(1500.0, 3000.0, (16, K)), dtype=torch.float32, device="cuda")
    ctx.surrogate_predict(q, p0)                       # mean 0, deviation 1
    half = n // 2                                      # (one call's pairs take slots of their own)
    for a, b in ((0, half), (half, n)):
        ctx.surrogate_add(torch.tensor(x[a:b], device="cuda"), torch.tensor(f[a:b], device="cuda"))
    for _ in range(50):
        ctx.surrogate_train(0, 16)                     # the statistics alone
        ctx.surrogate_predict(q, p1)
    y = np.log(f).astype(np.float32).astype(np.float64)
    if n > cap:                                        # the ring's oldest pairs are gone
        y = y[n - cap:]
    var = np.mean(y * y) - np.mean(y) ** 2 if n > 1 else 1.0
    sd, mu = np.sqrt(max(var, 1e-12)), np.mean(y)
    # two FP32 roundings (the deviation's and the mean's) and a product and a sum in FP32
    want = p0.cpu().numpy().astype(np.float64) * sd + mu
    tol = 4 * 2.0 ** -24 * (np.abs(p0.cpu().numpy()) * sd + abs(mu))
    assert np.all(np.abs(p1.cpu().numpy() - want) <= tol)
    assert ctx.device_error() == 0
    ctx.close()
