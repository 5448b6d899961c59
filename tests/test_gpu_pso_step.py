"""The swarm step's ranks by counting and its global best, over swarm sizes at
the edges of a warp, a CTA and the kernel's range, with tied, infinite and
not-a-number fitnesses, against numpy's stable sort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,D", [(2, 4), (7, 6), (8, 33), (33, 4), (257, 5), (1024, 8), (2047, 4), (2048, 4)])
def test_order_and_best(P, D):
    from paper_1905_12795_gb300 import binding as B
    from paper_1905_12795_gb300 import synth
    ctx = B.Context([B.make_grid(41, 41, 10.0, 10.0, 5, 4, 0.2, 10.0, 1500.0, 3000.0)],
                    synth.receiver_line(41, 10.0, 20.0), B.EmpsoPso(P, D, 1.2, 2.9, 0.5, 0.3, 0.5, 1, 1, 7), 0.0, 1.0)
    rng = np.random.default_rng(P)
    ctx.pso_init()
    x = torch.zeros(P, D, dtype=torch.float64, device="cuda")
    ctx.pso_get_state(x=x)
    x0 = x.cpu().numpy().copy()
    f = np.round(rng.normal(size=P), 1)                # many ties, both signs, both zeros
    f[rng.random(P) < 0.1] = np.inf
    f[rng.random(P) < 0.1] = np.nan
    f[rng.random(P) < 0.1] = -0.0
    ctx.pso_step(torch.tensor(f, device="cuda"))
    s = dict(p=torch.zeros_like(x), pf=torch.zeros(P, dtype=torch.float64, device="cuda"),
             order=torch.zeros(P, dtype=torch.int32, device="cuda"), gk=torch.zeros(2, dtype=torch.int32, device="cuda"))
    ctx.pso_get_state(**s)
    s = {k: v.cpu().numpy() for k, v in s.items()}
    key = np.where(np.isfinite(f), f, np.inf)
    assert np.array_equal(s["order"], np.argsort(key, kind="stable"))
    assert np.array_equal(s["pf"], key)
    assert s["gk"].tolist() == [int(np.argmin(key)), 1]
    done = np.isfinite(key)
    assert np.array_equal(s["p"][done], x0[done])
    ctx.close()
