"""Short windows: the low-pass that forms its taps in every CTA gives the bits of the
one that reads them from a table.  The same record once (few taps formed: no table) and
repeated until the call takes the table; each output is one sum in one order on both
paths."""
import pytest

from paper_1905_12795_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPAN, COLS, TAPS = 256, 256, 1 << 20       # the rule's limits


@pytest.mark.parametrize("nt_in,nrec,ratio,half", [(7, 3, 1.0, 0.5), (50, 40, 0.5, 1.0), (256, 257, 1.0, 2.0),
                                                   (300, 101, 3.7, 0.02), (300, 1, 10.0, 0.02), (1001, 7, 2.0, 0.05)])
def test_narrow_equals_table(nt_in, nrec, ratio, half):
    from paper_1905_12795_gb300 import binding as B
    ctx = B.Context([B.make_grid(61, 41, 10.0, 10.0, 10, 8, 0.25, 15.0, 1500.0, 3000.0)],
                    synth.receiver_line(61, 10.0, 20.0))
    dt, nt_out = 0.001, max(1, int(nt_in / ratio))
    span = min(nt_in, int((7 * dt * ratio + 2 * half) / dt) + 3)
    assert span <= SPAN and nt_out * span * -(-nrec // COLS) <= TAPS
    copies = (TAPS // (nt_out * span) + 1) * COLS // nrec + 1
    gen = torch.Generator(device="cuda").manual_seed(nt_in)
    x = torch.randn(1, nt_in, nrec, device="cuda", generator=gen)
    one, many = torch.zeros(1, nt_out, nrec, device="cuda"), torch.zeros(copies, nt_out, nrec, device="cuda")
    ctx.lowpass(x, dt, one, dt * ratio, 20.0, half)
    ctx.lowpass(x.expand(copies, -1, -1).contiguous(), dt, many, dt * ratio, 20.0, half)
    assert torch.isfinite(one).all() and one.abs().max() > 0
    assert torch.equal(many, one.expand_as(many))
    ctx.close()
