"""The low-pass's workspace: a context's first call finds it made, calls on other
streams than the first one's take memory of their own, a captured call leaves a
graph that may be cloned and used as a child."""
import ctypes
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


@pytest.mark.parametrize("big", [False, True])
def test_captured_call_in_clones_and_children(big):
    """A captured call replayed from the graph, from a clone after the graph is
    destroyed and from a child of another graph, with direct calls and further
    captures in between: the bits of direct calls."""
    rt = ctypes.CDLL("libcudart.so.13")
    V = ctypes.c_void_p

    def ok(rc):
        assert rc == 0, rc

    ctx = _ctx()
    args, out = _call(2, 8000, 461, 8000, 0.5, 4) if big else _call(seed=4)
    other, _ = _call(2, 3000, 100, 3000, 0.4, 5)
    x = args[0]
    st = torch.cuda.Stream()

    def capture(a):
        graph = V()
        ok(rt.cudaStreamBeginCapture(V(st.cuda_stream), 0))
        with torch.cuda.stream(st):
            ctx.lowpass(*a)
        ok(rt.cudaStreamEndCapture(V(st.cuda_stream), ctypes.byref(graph)))
        return graph

    def direct(a, o):
        o.zero_()
        ctx.lowpass(*a)
        torch.cuda.synchronize()
        return o.cpu().numpy().copy()

    direct(args, out)                       # the kernels are loaded
    graph = capture(args)
    clone, parent, node = V(), V(), V()
    ok(rt.cudaGraphClone(ctypes.byref(clone), graph))
    ok(rt.cudaGraphCreate(ctypes.byref(parent), 0))
    ok(rt.cudaGraphAddChildGraphNode(ctypes.byref(node), parent, None, ctypes.c_size_t(0), graph))
    execs = []
    for g in (graph, clone, parent):
        e = V()
        ok(rt.cudaGraphInstantiate(ctypes.byref(e), g, ctypes.c_ulonglong(0)))
        ok(rt.cudaGraphDestroy(g))
        execs.append(e)
    for k in range(4):
        x.copy_(torch.randn_like(x))
        want = direct(args, out)
        ok(rt.cudaGraphDestroy(capture(other)))          # another table, taken and given back
        direct(other, other[2])
        for e in execs:
            out.zero_()
            torch.cuda.synchronize()
            ok(rt.cudaGraphLaunch(e, V(st.cuda_stream)))
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), want)
    for e in execs:
        ok(rt.cudaGraphExecDestroy(e))
    ctx.close()
