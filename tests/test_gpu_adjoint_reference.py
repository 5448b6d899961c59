"""The gradient at the edge sizes of the persistent backward pass against FP64.

The reference is the scheme in torch's FP64 with its derivative by automatic
differentiation, and its traces are first compared with the oracle's.  A few shots
each, so that one launch's groups hold all instances (`persistent` restates when they
do): odd widths with a ragged last column group, rows of one run, a grid narrower
than a warp, sources and receivers off the nodes, sharing a cell, and at the corners.

Bound, derived before the first run: a step rounds u^{n+1} by about 4 2^-24 of it, and
a leapfrog carries a step's error on in proportion to the steps that follow, so a field
is off by at most 4 2^-24 nt^2 / 2 of its size, and the gradient, a product of two
fields, by twice that.
"""
import numpy as np
import pytest

import oracle
from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DT, NT = 2.0 ** -10, 60


def persistent(nx, nz, pad, order, S):
    """Does the backward pass of S shots run as one launch on groups of CTAs?"""
    prop = torch.cuda.get_device_properties(0)
    threads, ctas = 128, 2 * prop.multi_processor_count
    NZ, NQ = nz + 2 * pad, (nx + 2 * pad + 3) // 4
    room = prop.shared_memory_per_block_optin // 2 - (12 << 10)
    for flight in range(1 if order == 16 else S, S + 1):
        runs = min(NZ, (ctas // flight - 1) * threads // NQ)
        if runs >= 1 and 48 * -(-NZ // runs) * threads <= room:
            return True
    return False


def reference(og, vel, shots, rec, dobs):
    """(traces [S][nt][nrec], gradient of 1/2 sum (traces - dobs)^2 by vel) in FP64."""
    f64 = dict(dtype=torch.float64)
    c = oracle.fd_coeffs(og.order)
    R, pad = len(c) - 1, og.pad
    NX, NZ = og.nx + 2 * pad, og.nz + 2 * pad

    def weights(xz):
        w = torch.zeros(len(xz), NZ, NX, **f64)
        for k, (x, z) in enumerate(xz):
            fx, fz = x / og.hx + pad, z / og.hz + pad
            i, j = min(int(fx), NX - 2), min(int(fz), NZ - 2)
            ax, az = fx - i, fz - j
            for dj, di, q in ((0, 0, (1 - ax) * (1 - az)), (0, 1, ax * (1 - az)), (1, 0, (1 - ax) * az), (1, 1, ax * az)):
                w[k, j + dj, i + di] += q
        return w

    src, at = weights(shots) / (og.hx * og.hz), weights(rec).reshape(len(rec), -1)
    t = (torch.tensor(oracle.damping_profile(og.nx, pad, og.hx, og.vmax))[None, :]
         + torch.tensor(oracle.damping_profile(og.nz, pad, og.hz, og.vmax))[:, None]) * (og.dt / 2)
    r = oracle.ricker(og.f0, np.arange(og.nt) * og.dt)
    v = torch.tensor(vel, requires_grad=True, **f64)
    a = torch.nn.functional.pad(v[None, None], (pad,) * 4, mode="replicate")[0, 0] ** 2 * og.dt ** 2

    def lap(u):
        p = torch.nn.functional.pad(u, (R,) * 4)
        out = c[0] * (1 / og.hx ** 2 + 1 / og.hz ** 2) * u
        for m in range(1, R + 1):
            out = out + c[m] / og.hx ** 2 * (p[:, R:R + NZ, R - m:R - m + NX] + p[:, R:R + NZ, R + m:R + m + NX])
            out = out + c[m] / og.hz ** 2 * (p[:, R - m:R - m + NZ, R:R + NX] + p[:, R + m:R + m + NZ, R:R + NX])
        return out

    prev = cur = torch.zeros(len(shots), NZ, NX, **f64)
    traces = []
    for n in range(og.nt):
        prev, cur = cur, (2 * cur - (1 - t) * prev + a * (lap(cur) + r[n] * src)) / (1 + t)
        traces.append(cur.reshape(len(shots), -1) @ at.T)
    traces = torch.stack(traces, 1)
    (0.5 * ((traces - dobs) ** 2).sum()).backward()
    return traces.detach().numpy(), v.grad.numpy()


SIZES = [(150, 61, 20, 8, 4), (33, 90, 5, 4, 3), (401, 30, 3, 2, 5), (61, 40, 11, 16, 3), (9, 30, 3, 8, 2), (30, 9, 0, 16, 2)]


def problem(nx, nz, pad, order, S):
    h = 10.0
    og = oracle.Grid(nx, nz, h, h, pad, order, (NT - 1) * DT, 60.0, 3200.0, dt=DT)
    assert og.nt == NT
    vel = synth.layered_faulted_model(nx, nz, h, h, seed=3, vmin=1500.0, vmax=3000.0).astype(np.float32).astype(np.float64)
    X, Z = (nx - 1) * h, (nz - 1) * h
    shots = np.array([[16.0 * np.floor(X * (k + 0.5) / S / 16.0) + 3.25, 8.0 * np.floor(Z * k / S / 8.0) + 2.125]
                      for k in range(S)])
    line = np.array([[10.0 * i + 1.25, 12.5] for i in range(nx - 1)])
    rec = np.concatenate([line, line[::3] + [2.0, 1.5], [[0.0, 0.0], [X, 0.0], [0.0, Z], [X, Z], [X - 1.25, Z - 1.25]]])
    gen = torch.Generator().manual_seed(nx)
    dobs = (1e-4 * torch.randn(S, NT, len(rec), generator=gen)).double()
    return og, vel, shots, rec, dobs


@pytest.mark.parametrize("nx,nz,pad,order,S", SIZES)
def test_gradient_against_fp64(nx, nz, pad, order, S):
    from paper_1905_12795_gb300 import binding as B
    assert persistent(nx, nz, pad, order, S)
    og, vel, shots, rec, dobs = problem(nx, nz, pad, order, S)
    n = len(rec)
    traces, ref = reference(og, vel, shots, rec, dobs)
    _, want = oracle.shot_batch(og, vel, shots, rec, [0] * S, [n] * S, want_traces=True)
    assert np.abs(traces - np.stack(want)).max() <= 1e-10 * np.abs(traces).max()
    ctx = B.Context([B.make_grid(nx, nz, og.hx, og.hz, pad, order, og.T, og.f0, 1500.0, og.vmax, dt=DT)], rec)
    assert ctx.grid_info(0)[1] == NT
    grad = torch.zeros(1, nz, nx, device="cuda")
    ctx.gradient(torch.tensor(vel[None], dtype=torch.float32, device="cuda"), B.make_shots(shots, [0] * S, [n] * S),
                 dobs.float().cuda().reshape(-1), grad)
    got = grad[0].cpu().double().numpy()
    assert ctx.device_error() == 0
    ctx.close()
    assert np.linalg.norm(got - ref) <= 4 * NT ** 2 * 2.0 ** -24 * np.linalg.norm(ref)
