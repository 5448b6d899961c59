"""The low-pass kernel's tiles against the oracle: column counts at the edges
of every tile width, output counts around a tile, sparse outputs (a step far
beyond the window), and input samples that are not numbers, which reach only
the outputs of the groups of 8 whose window holds them."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(x, dt_in, nt_out, dt_out, fc, W):
    from paper_1905_12795_gb300 import binding as B
    ctx = B.Context([B.make_grid(11, 11, 10.0, 10.0, 0, 2, 0.05, 10.0, 1500.0, 2000.0)], [[0.0, 0.0]])
    out = torch.full((x.shape[0], nt_out, x.shape[2]), 7.0, device="cuda")
    ctx.lowpass(torch.tensor(x, device="cuda"), dt_in, out, dt_out, fc, W)
    got = out.cpu().numpy()
    ctx.close()
    return got


@pytest.mark.parametrize("S,nt_in,nrec,nt_out,dt_out,W", [
    (1, 300, 1, 31, 2e-3, 0.05), (1, 300, 33, 33, 2e-3, 0.05), (3, 211, 85, 64, 2e-3, 0.08),
    (5, 400, 461, 97, 2.3e-3, 0.03), (16, 1500, 461, 700, 2.1e-3, 0.04),
    (2, 900, 40, 12, 7e-2, 0.02), (2, 20, 500, 9, 1e-3, 0.5)])
def test_tiles_match_oracle(S, nt_in, nrec, nt_out, dt_out, W):
    x = np.random.default_rng(nt_in + nrec).normal(size=(S, nt_in, nrec)).astype(np.float32)
    got = _run(x, 1e-3, nt_out, dt_out, 20.0, W)
    ref = oracle.lowpass(x.astype(np.float64), 1e-3, nt_out, dt_out, 20.0, W)
    for s in range(S):      # FP32 taps and sums of a few hundred products, as in the other parity test
        assert np.max(np.abs(got[s] - ref[s])) < 2e-5 * max(np.max(np.abs(ref[s])), 1e-30)


def test_not_a_number_stays_in_its_groups():
    x = np.random.default_rng(1).normal(size=(1, 400, 5)).astype(np.float32)
    clean = _run(x, 1e-3, 200, 2e-3, 20.0, 0.03)
    x[0, 200, 2] = np.nan
    got = _run(x, 1e-3, 200, 2e-3, 20.0, 0.03)
    hit = ~np.isfinite(got[0])
    assert not hit[:, [0, 1, 3, 4]].any()
    # groups of 8 outputs (16 ms) whose window of 30 ms either side holds t = 200 ms
    first, last = 0.002 * 8 * np.arange(25), 0.002 * (8 * np.arange(25) + 7)
    holds = np.repeat((first - 0.03 <= 0.2) & (last + 0.03 >= 0.2), 8)
    assert np.array_equal(hit[:, 2], holds)
    assert np.array_equal(got[0][~hit], clean[0][~hit])
