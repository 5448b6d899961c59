"""The low-pass's workspace: a context's first call finds it made, calls on other
streams than the first one's take memory of their own."""
import time

import numpy as np
import pytest

from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ctx():
    from paper_1905_12795_gb300 import binding as B
    return B.Context([B.make_grid(61, 41, 10.0, 10.0, 10, 8, 0.2, 15.0, 1500.0, 3000.0)],
                     synth.receiver_line(61, 10.0, 20.0))


def _call(S=1, nt=300, R=40, nt_out=150, half=0.1, seed=0):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(S, nt, R, device="cuda", generator=gen)
    out = torch.zeros(S, nt_out, R, device="cuda")
    return (x, 0.002, out, 0.002 * (nt - 1) / (nt_out - 1), 10.0, half), out


def test_first_call_of_a_context_is_no_set_up():
    """Host time of a short record's first call less that of the later ones (a pool
    created and mapped in it took 140 us, the kernels take 35)."""
    args, _ = _call()
    extra = []
    for i in range(9):
        ctx = _ctx()
        torch.cuda.synchronize()
        t = []
        for _ in range(8):
            t0 = time.perf_counter()
            ctx.lowpass(*args)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        if i:                               # (the process's first call loads the kernels)
            extra.append(t[0] - min(t[1:]))
        ctx.close()
    assert min(extra) < 80e-6, extra


def test_streams_do_not_share_a_workspace():
    """Long calls enqueued on three streams of one context at once, with other
    parameters each: the same bits as one after the other."""
    ctx = _ctx()
    calls = [_call(4, 2000, 300, 1500, 0.3, 1), _call(4, 2000, 300, 500, 0.5, 2), _call(1, 20000, 461, 20000, 1.0, 3)]
    ref = []
    for args, out in calls:
        ctx.lowpass(*args)
        ref.append(out.cpu().numpy().copy())
    streams = [torch.cuda.Stream() for _ in calls]
    for _ in range(10):
        for _, out in calls:
            out.zero_()
        torch.cuda.synchronize()
        for st, (args, _) in zip(streams, calls):
            with torch.cuda.stream(st):
                ctx.lowpass(*args)
        torch.cuda.synchronize()
        for r, (_, out) in zip(ref, calls):
            assert np.array_equal(out.cpu().numpy(), r)
    ctx.close()
