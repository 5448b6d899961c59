"""Misfits of the plain streaming kernel (order 16, mixed orders, the
allocation-free entry point): squares of the FP32 residuals and their sums are
held in FP64 (the L2 kernel's in FP32 over 32 steps of one receiver), so residuals whose squares leave FP32's range keep a finite
misfit, and no split of the GPU changes it by more than FP64 rounding."""
import numpy as np
import pytest

from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# A sum of N squares (each exact in FP64) in any order: relative error below N 2^-53;
# N = shots x receivers x steps stays below 2^22 here, and the reference sum has as many
TOL = 2.0 ** -30
BIG = float(np.float32(3e19))           # its square is past FP32; absorbs the traces (|d| << ulp)


@pytest.fixture(scope="module")
def B():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1905_12795_gb300 import binding
    binding.load()
    return binding


def _setup(B, orders, nrec, S, nx=61, nz=41, h=10.0):
    grids = [B.make_grid(nx, nz, h, h, 10, o, 0.1, 15.0, 1500.0, 3200.0, kx=4, kz=3) for o in orders]
    line = synth.receiver_line(nx, h, 1.25 * h)
    rec = np.tile(line, (-(-nrec // len(line)), 1))[:nrec]
    xz = synth.shot_line(S, (nx - 1) * h, 1.5 * h)
    return grids, rec, xz


@pytest.mark.parametrize("nrec,S", [(61, 1), (461, 2), (1300, 40)])
def test_order16_misfit_is_the_fp64_sum_of_its_traces(B, nrec, S):
    grids, rec, xz = _setup(B, [16], nrec, S)
    ctx = B.Context(grids, rec)
    nt = ctx.grid_info(0)[1]
    shots = B.make_shots(xz, [0] * S, [nrec] * S)
    vel = torch.tensor(synth.layered_faulted_model(61, 41, 10.0, 10.0, seed=3, vmin=1500.0, vmax=3200.0),
                       dtype=torch.float32, device="cuda")[None].contiguous()
    d = torch.zeros(S, nt, nrec, device="cuda")
    ctx.forward_traces(vel, shots, d)
    gen = torch.Generator(device="cuda").manual_seed(nrec)
    mis = torch.zeros(1, dtype=torch.float64, device="cuda")
    for dobs in (0.3 * d.std() * torch.randn(S, nt, nrec, device="cuda", generator=gen), torch.full_like(d, BIG)):
        ctx.eval_models(vel, shots, dobs.contiguous(), mis)
        want = 0.5 * ((d - dobs).double() ** 2).sum().item()
        assert np.isfinite(want) and abs(mis.item() - want) <= TOL * want
    assert ctx.device_error() == 0
    ctx.close()


def test_mixed_orders_keep_large_residuals(B):
    nrec, S, P = 300, 2, 3
    grids, rec, xz = _setup(B, [16, 4], nrec, S)
    ctx = B.Context(grids, rec)
    nts = [ctx.grid_info(i)[1] for i in range(2)]
    shots = B.make_shots(np.concatenate([xz, xz]), [0] * 4, [nrec] * 4, grid_ids=[0, 0, 1, 1])
    n = S * nrec * sum(nts)
    x = torch.tensor(synth.random_particles(P, 12, 1500.0, 3200.0, seed=4), dtype=torch.float32, device="cuda")
    mis = torch.zeros(P, dtype=torch.float64, device="cuda")
    ctx.eval_fitness(x, shots, torch.full((n,), BIG, device="cuda"), mis)
    assert ctx.last_launch()[0] == 1
    want = 0.5 * n * BIG * BIG
    assert np.all(np.abs(mis.cpu().numpy() - want) <= TOL * want)
    ctx.close()


@pytest.mark.parametrize("order", [2, 4, 8, 16])
def test_allocation_free_misfit_keeps_large_residuals(B, order):
    nrec, S = 300, 2
    grids, rec, xz = _setup(B, [order], nrec, S)
    nt = B.time_axis(grids[0])[1]
    n = S * nrec * nt
    mis = torch.zeros(1, dtype=torch.float64, device="cuda")
    vel = torch.full((1, 41, 61), 2000.0, device="cuda")
    B.eval_models_noalloc(grids[0], rec, vel, B.make_shots(xz, [0] * S, [nrec] * S),
                          torch.full((n,), BIG, device="cuda"), mis)
    want = 0.5 * n * BIG * BIG
    assert abs(mis.item() - want) <= TOL * want


def test_l2_misfit_sums_32_steps_of_one_receiver_in_fp32(B):
    """The L2 kernel's FP32 sums: 32 squares of 6e36 fit FP32, 64 do not, so no
    thread may add two receivers into one (64 shots of 1500 receivers give a
    thread two)."""
    nrec, S, c2 = 1500, 64, 6e36
    grids, rec, xz = _setup(B, [8], nrec, S)
    ctx = B.Context(grids, rec)
    nt = ctx.grid_info(0)[1]
    ctx.set_kernel(3)
    big = float(np.float32(np.sqrt(c2)))
    mis = torch.zeros(1, dtype=torch.float64, device="cuda")
    ctx.eval_models(torch.full((1, 41, 61), 2000.0, device="cuda"), B.make_shots(xz, [0] * S, [nrec] * S),
                    torch.full((S, nt, nrec), big, device="cuda"), mis)
    assert ctx.last_launch()[0] == 3 and nt > 64
    want = 0.5 * S * nt * nrec * big * big
    assert abs(mis.item() - want) <= 32 * 2.0 ** -24 * want       # 32 FP32 additions
    ctx.close()
