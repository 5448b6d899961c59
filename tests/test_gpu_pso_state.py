"""The swarm's state in one launch, by one copy (a single buffer) and by copies (the
largest swarms): the same values on every path, and nothing written past them."""
import pytest

from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,D", [(7, 3), (1024, 1024), (2048, 513)])
def test_paths_agree(P, D):
    from paper_1905_12795_gb300 import binding as B
    ctx = B.Context([B.make_grid(61, 41, 10.0, 10.0, 10, 8, 0.25, 15.0, 1500.0, 3000.0)],
                    synth.receiver_line(61, 10.0, 20.0), B.EmpsoPso(P, D, 1.2, 2.9, 0.5, 0.3, 0.25, 1, 1, 7), 1500.0, 3000.0)
    gen = torch.Generator(device="cuda").manual_seed(P)
    f64 = dict(dtype=torch.float64, device="cuda")
    given = {k: torch.rand(P, D, generator=gen, **f64) for k in ("x", "v", "p")}
    given["pf"] = torch.rand(P, generator=gen, **f64)
    ctx.pso_set_state(*given.values(), 5, 9)
    given["gk"] = torch.tensor([5, 9], dtype=torch.int32, device="cuda")

    def room(name):
        t = given[name]
        return torch.full((t.numel() + 2,), -1, dtype=t.dtype, device="cuda")

    whole = {k: room(k) for k in given}
    ctx.pso_get_state(**whole)
    for k, t in given.items():
        alone = room(k)
        ctx.pso_get_state(**{k: alone})
        for got in (whole[k], alone):
            assert torch.equal(got[:-2], t.reshape(-1)) and bool((got[-2:] == -1).all())
    ctx.close()
