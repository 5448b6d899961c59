"""Grids whose wavefield buffer holds more than 4 GB, where a 32-bit byte offset
wraps: source and receivers in the last rows, past the 4 GB line, against a small
grid with the same corner of the model.  The waves (and the stencils' reach over
all steps) stay clear of the sides where the two grids differ, every coordinate
is a multiple of a power of two, and a point's arithmetic does not depend on the
split of the GPU: the traces are the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NX, NZ, H, NT = 16384, 65600, 8.0, 24          # 65616 rows of 16416 floats: 4.3 GB


@pytest.mark.parametrize("order,kind", [(16, 0), (8, 3)])
def test_traces_past_4_gb(order, kind):
    from paper_1905_12795_gb300 import binding as B
    assert (NZ + 16) * (NX + 32) > 2 ** 30
    reach = 2 * NT * order // 2                 # there and back
    nx, nz = 64 + reach + 64, 64 + reach + 64
    dt = 0.0008
    corner = torch.tensor(np.random.default_rng(order).uniform(1500.0, 3200.0, (nz, nx)), dtype=torch.float32,
                          device="cuda")
    up = 20                                     # rows above the bottom
    rec = np.stack([np.arange(30, 96) * H, np.full(66, up * H - 4.0)], 1)      # from the bottom
    got = []
    for gx, gz in ((nx, nz), (NX, NZ)):
        vel = torch.full((1, gz, gx), 2000.0, device="cuda")
        vel[0, -nz:, :nx] = corner
        bottom = (gz - 1) * H
        ctx = B.Context([B.make_grid(gx, gz, H, H, 0, order, (NT - 1) * dt, 30.0, 1500.0, 3200.0, kx=2, kz=2, dt=dt)],
                        np.stack([rec[:, 0], bottom - rec[:, 1]], 1))
        assert ctx.grid_info(0)[1] == NT
        ctx.set_kernel(kind)
        out = torch.zeros(1, NT, len(rec), device="cuda")
        ctx.forward_traces(vel, B.make_shots([[62 * H, bottom - (up + 2) * H]], [0], [len(rec)]), out)
        assert ctx.last_launch()[0] == (3 if kind == 3 else 1)
        assert ctx.device_error() == 0
        got.append(out.cpu().numpy())
        ctx.close()
        del vel
    torch.cuda.empty_cache()
    assert np.abs(got[0]).max() > 0 and np.array_equal(*got)
