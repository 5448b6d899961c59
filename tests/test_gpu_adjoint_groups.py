"""The persistent backward pass against the per-step kernels at the sizes where
its split can go wrong.  Up to order 8, more instances than one round holds run
step by step, so a batch's gradient must equal the sum of its shots' gradients
taken one at a time (FP32 sums over the shots in another order); odd widths (a
ragged last column group), receivers sharing a cell and off the nodes, rows of
one run, and a grid narrower than a warp."""
import numpy as np
import pytest

from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,pad,order,S", [(150, 61, 20, 8, 70), (33, 90, 5, 4, 160), (401, 30, 3, 2, 60),
                                               (61, 40, 11, 16, 5), (9, 30, 3, 8, 3)])
def test_batch_equals_its_shots(nx, nz, pad, order, S):
    from paper_1905_12795_gb300 import binding as B
    h, T = 10.0, 0.12
    rec = np.concatenate([synth.receiver_line(nx, h, 1.25 * h), synth.receiver_line(nx, h, 1.25 * h)[:-1] + [3.3, 2.1]])
    nrec = len(rec)
    ctx = B.Context([B.make_grid(nx, nz, h, h, pad, order, T, 20.0, 1500.0, 3200.0)], rec)
    nt = ctx.grid_info(0)[1]
    vel = torch.tensor(synth.layered_faulted_model(nx, nz, h, h, seed=3, vmax=3000.0), dtype=torch.float32,
                       device="cuda")[None].contiguous()
    xz = synth.shot_line(S, (nx - 1) * h, 1.4 * h)
    gen = torch.Generator(device="cuda").manual_seed(nx)
    d = 0.1 * torch.randn(S, nt * nrec, device="cuda", generator=gen)
    whole, one = torch.zeros(1, nz, nx, device="cuda"), torch.zeros(1, nz, nx, device="cuda")
    ctx.gradient(vel, B.make_shots(xz, [0] * S, [nrec] * S), d.reshape(-1), whole)
    total, size = torch.zeros(1, nz, nx, dtype=torch.float64, device="cuda"), 0.0
    for s in range(S):
        ctx.gradient(vel, B.make_shots(xz[s:s + 1], [0], [nrec]), d[s].contiguous(), one)
        total += one.double()
        size += float(one.double().norm())
    assert ctx.device_error() == 0
    # FP32 sums over S shots: half an ulp of a partial sum each
    assert float((whole.double() - total).norm()) <= S * 2.0 ** -24 * size
    ctx.close()
