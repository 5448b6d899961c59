"""Gradients of two contexts on two host threads and streams, one of a grid whose
backward pass takes much shared memory, one of a small grid whose pass takes
little: the kernel's limit is the process's, and neither thread may lower it
between the other's split and its launch.  Nearly every call captures a new graph."""
import threading

import numpy as np
import pytest

from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Case:
    def __init__(self, nx, nz, order, least):
        from paper_1905_12795_gb300 import binding as B
        h = 10.0
        rec = synth.receiver_line(nx, h, 1.25 * h)
        self.ctx = B.Context([B.make_grid(nx, nz, h, h, 5, order, 0.02, 20.0, 1500.0, 3200.0)], rec)
        nt = self.ctx.grid_info(0)[1]
        self.vel = torch.tensor(synth.layered_faulted_model(nx, nz, h, h, seed=3, vmax=3000.0), dtype=torch.float32,
                                device="cuda")[None].contiguous()
        gen = torch.Generator(device="cuda").manual_seed(nx)
        self.d = torch.randn((least + 5) * nt * nx, device="cuda", generator=gen)
        self.shots = [B.make_shots(synth.shot_line(S, (nx - 1) * h, 1.4 * h), [0] * S, [nx] * S) for S in range(least, least + 6)]
        self.grad = torch.zeros(1, nz, nx, device="cuda")
        self.first, self.worst, self.error = {}, 0.0, None
        self.call(0)                        # everything loaded and allocated before the threads start

    def call(self, n):
        s = n % 6
        self.ctx.set_gradient_chains(n // 6 % 9)       # (the number is part of a graph's key)
        self.ctx.gradient(self.vel, self.shots[s], self.d, self.grad)
        g = self.grad.cpu().numpy()
        ref = self.first.setdefault(s, g)
        self.worst = max(self.worst, np.linalg.norm(g - ref) / np.linalg.norm(ref))

    def loop(self, calls, stop):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                n = 0
                while n < calls and not stop.is_set():
                    self.call(n)
                    n += 1
        except Exception as e:              # noqa: BLE001 - reported by the main thread
            self.error = e
        stop.set()


@pytest.mark.parametrize("order", [8, 16])
def test_two_threads_two_sizes(order):
    for _ in range(2):
        # (rows of the big grid's threads: about 12 with so many shots in flight, over 48 KB)
        big, small, stop = Case(401, 151, order, 10), Case(33, 21, order, 1), threading.Event()
        torch.cuda.synchronize()
        threads = [threading.Thread(target=big.loop, args=(54, stop)), threading.Thread(target=small.loop, args=(10 ** 9, stop))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for c in (big, small):
            assert c.error is None, c.error
            assert c.ctx.device_error() == 0
            # (receivers of one cell are added atomically: last bits may differ)
            assert c.worst <= 1e-4
            c.ctx.close()
