"""GPU: dequantizing more states than are resident at once (they leave by bulk stores from shared memory, where two CTAs fit on an SM
so) against the same states a few at a time.  One state more than that, several to a CTA, windows that just fit and just do not."""
import pytest
import torch

from paper_2609_38166_b200 import lq, synth

pytestmark = pytest.mark.gpu

G, K = synth.GATE_SCALAR, synth.GATE_DIAG


@pytest.mark.parametrize("gate,batch,heads,W,r,rec16", [(G, 99, 3, 16, 4, 0), (K, 99, 3, 16, 4, 0), (K, 100, 8, 17, 8, 0), (G, 100, 8, 24, 4, 0), (G, 75, 4, 25, 4, 0),
                                                        (G, 120, 4, 9, 1, 1), (K, 75, 4, 13, 3, 1), (G, 1200, 1, 1, 16, 0), (K, 150, 2, 64, 2, 0)])
def test_many_states_and_few_at_a_time_give_the_same_bits(gate, batch, heads, W, r, rec16):
    shape = lambda n: lq.Shape(n, heads, heads, 128, 128, W, r, 1, gate, 1, 1, rec16, 0)
    gen = torch.Generator("cuda").manual_seed(W + r)
    st = lq.State(shape(batch))
    lq.quantize_state(shape(batch), torch.randn((batch, heads, 128, 128), generator=gen, device="cuda"), st)
    st.records.copy_(torch.rand(st.records.shape, generator=gen, device="cuda") * 0.8 + 0.1)
    st.decays.copy_(torch.rand(st.decays.shape, generator=gen, device="cuda") * 0.8 + 0.1)
    st.win_pos.copy_(torch.arange(batch, device="cuda") % (W + 1))
    S = torch.full((batch + 1, heads, 128, 128), 7.0, device="cuda")
    lq.dequantize_state(shape(batch), st, S[:batch])
    step = 64 // heads
    for b in range(0, batch, step):
        n = min(step, batch - b)
        part, out = lq.State(shape(n)), torch.zeros((n, heads, 128, 128), device="cuda")
        for name in ("heads", "records", "decays", "win_pos"):
            getattr(part, name).copy_(getattr(st, name)[b:b + n])
        lq.dequantize_state(shape(n), part, out)
        assert torch.equal(out, S[b:b + n]), b
    assert (S[batch] == 7.0).all() and lq.check_device() == 0
