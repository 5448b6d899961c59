"""The plain streaming kernel on groups of co-resident CTAs, at the sizes where
its split can go wrong: rows shorter than a warp (several runs in one warp),
rows one group past a warp, runs of one row (more threads than the grid has
rows to give), a grid of several rounds of instances, two stencil radii in one
launch, and order 16 through the gradient's forward pass."""
import numpy as np
import pytest

import oracle
from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TRACE_TOL = 1e-4        # relative l2 of a shot's traces, as in the other parity tests


@pytest.fixture(scope="module")
def B():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1905_12795_gb300 import binding
    binding.load()
    return binding


def _dev(a, dtype=torch.float32):
    return torch.tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _case(nx, nz, h, pad, order, S, T=0.2, f0=15.0, vmax=3200.0):
    og = oracle.Grid(nx, nz, h, h, pad, order, T, f0, vmax)
    vel = synth.layered_faulted_model(nx, nz, h, h, seed=nx + nz, vmin=1500.0, vmax=vmax)
    shots = synth.shot_line(S, (nx - 1) * h, 1.5 * h) + np.array([0.3 * h, 0.0])
    shots[:, 0] = np.minimum(shots[:, 0], (nx - 1) * h)
    rec = synth.receiver_line(nx, h, 1.25 * h)
    return og, vel, shots, rec


# columns: 3 groups (ten runs in a warp), 8 + 25 = 33 groups, 128 = a CTA, 261; rows down to 6
@pytest.mark.parametrize("nx,nz,pad,S", [(5, 90, 2, 2), (5, 6, 2, 1), (113, 21, 9, 1), (512, 9, 0, 2),
                                         (401, 40, 12, 3), (61, 40, 11, 40)])
def test_order16_traces_at_edge_sizes(B, nx, nz, pad, S):
    og, vel, shots, rec = _case(nx, nz, 10.0, pad, 16, S)
    nrec = len(rec)
    _, ref = oracle.shot_batch(og, vel, shots, rec, [0] * S, [nrec] * S, want_traces=True)
    ctx = B.Context([B.make_grid(nx, nz, 10.0, 10.0, pad, 16, 0.2, 15.0, 1500.0, 3200.0)], rec)
    out = torch.zeros(S, og.nt, nrec, device="cuda")
    ctx.forward_traces(_dev(vel[None]), B.make_shots(shots, [0] * S, [nrec] * S), out)
    got = out.cpu().numpy()
    for s in range(S):
        err = np.linalg.norm(got[s] - ref[s]) / np.linalg.norm(ref[s])
        assert err < TRACE_TOL, (s, err)
    assert ctx.device_error() == 0
    ctx.close()


def test_two_radii_in_one_launch(B):
    """Orders 16 and 4 on one generation's shots: the instances' misfits add up
    to those of each order by itself."""
    h, S = 10.0, 2
    _, vel, shots, rec = _case(61, 41, h, 10, 16, S)
    nrec = len(rec)
    grids = [B.make_grid(61, 41, h, h, 10, o, 0.2, 15.0, 1500.0, 3200.0, kx=4, kz=3) for o in (16, 4)]
    x = _dev(synth.random_particles(3, 12, 1500.0, 3200.0, seed=4))
    got = {}
    for ids in ((0,), (1,), (0, 1)):
        ctx = B.Context(grids, rec)
        n = sum(ctx.grid_info(i)[1] for i in ids) * S * nrec
        sh = B.make_shots(np.concatenate([shots] * len(ids)), [0] * S * len(ids), [nrec] * S * len(ids),
                          grid_ids=[i for i in ids for _ in range(S)])
        mis = torch.zeros(3, dtype=torch.float64, device="cuda")
        ctx.set_kernel(1 if ids == (1,) else 0)
        ctx.eval_fitness(x, sh, torch.zeros(n, device="cuda"), mis)
        assert ctx.device_error() == 0
        got[ids] = mis.cpu().numpy()
        ctx.close()
    assert np.allclose(got[(0, 1)], got[(0,)] + got[(1,)], rtol=1e-4)
