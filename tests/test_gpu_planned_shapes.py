"""A shape planned once is the one a fresh context plans, for batches of several sizes
and shots of several receiver counts in turn, also after a forced shape."""
import pytest

from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(B, ctx, nt, M, nrec):
    x = torch.tensor(synth.random_particles(M, 32, 1500.0, 3000.0, seed=M), dtype=torch.float32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(nrec)
    d = 0.1 * torch.randn(nt * nrec, device="cuda", generator=gen)
    mis = torch.zeros(M, dtype=torch.float64, device="cuda")
    ctx.eval_fitness(x, B.make_shots([[400.0, 20.0]], [0], [nrec]), d, mis)
    return ctx.last_launch(), ctx.last_tile_rows(), ctx.last_clusters(), mis


@pytest.mark.parametrize("order", [2, 8])
def test_same_as_a_fresh_context(order):
    from paper_1905_12795_gb300 import binding as B
    nx, nz, h = 91, 61, 10.0
    grid = B.make_grid(nx, nz, h, h, 15, order, 0.08, 25.0, 1500.0, 3200.0)
    rec = synth.receiver_line(nx, h, 20.0)
    ctx = B.Context([grid], rec)
    nt = ctx.grid_info(0)[1]
    for M, nrec in ((1, nx), (40, nx), (1, nx), (1, 5), (40, 5), (300, nx), (40, nx)):
        fresh = B.Context([grid], rec)
        want, got = _run(B, fresh, nt, M, nrec), _run(B, ctx, nt, M, nrec)
        assert got[:3] == want[:3] and torch.equal(got[3], want[3])
        ctx.set_cluster(4)
        assert _run(B, ctx, nt, M, nrec)[0][1] == 4
        ctx.set_cluster(0)
        fresh.close()
    ctx.close()
