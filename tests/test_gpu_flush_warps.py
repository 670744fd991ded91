"""GPU: the window boundary of many due heads at a time, where a state with four compensators, the scalar gate and fp32 records
is held by four warps, against the same heads a few at a time, which eight warps take.  Both record formats, both gates, one round
and two, lists of due sequences in one trip and in two, and calls of window_flush."""
import pytest
import torch

from paper_2609_38166_b200 import lq, synth

pytestmark = pytest.mark.gpu

G, K = synth.GATE_SCALAR, synth.GATE_DIAG


@pytest.mark.parametrize("gate,batch,heads,W,r,n_iter,rec16", [
    (G, 256, 32, 16, 4, 1, 0), (G, 256, 32, 16, 4, 1, 1), (K, 256, 32, 16, 4, 1, 0), (K, 256, 32, 16, 4, 1, 1), (G, 100, 32, 8, 4, 2, 0),
    (G, 256, 8, 6, 3, 1, 0), (K, 100, 24, 8, 8, 1, 0), (G, 1024, 5, 16, 4, 1, 0), (G, 1025, 5, 16, 4, 1, 0), (G, 1500, 4, 17, 4, 1, 1), (G, 2048, 3, 16, 4, 1, 0),
    (G, 2049, 3, 16, 4, 1, 0), (G, 37, 8, 1, 4, 1, 0), (G, 333, 1, 1, 4, 1, 0)])
def test_many_due_heads_and_few_at_a_time_give_the_same_bits(gate, batch, heads, W, r, n_iter, rec16):
    shape = lambda n: lq.Shape(n, heads, heads, 128, 128, W, r, n_iter, gate, 1, 1, rec16, 0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert batch * heads // W >= 2 * sms
    gen = torch.Generator("cuda").manual_seed(batch + W)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")
    whole, other = lq.State(shape(batch), work=False), lq.State(shape(batch), work=False)
    lq.quantize_state(shape(batch), normal(batch, heads, 128, 128), whole)
    for x in (whole.records, whole.decays):
        x.copy_(torch.rand(x.shape, generator=gen, device="cuda") * 0.8 + 0.1)
    few = max(1, 160 // heads)
    cuts = [slice(b, min(b + few, batch)) for b in range(0, batch, few)]
    parts = [lq.State(shape(c.stop - c.start), work=False, storage=tuple(t[c] for t in other.tensors())) for c in cuts]
    rank = torch.randperm(batch, generator=gen, device="cuda").to(torch.int32)
    last = torch.where(torch.arange(batch, device="cuda") == batch - 1, W - 1, 0).to(torch.int32)
    o = [torch.zeros((batch, heads, 128), device="cuda") for _ in range(2)]

    def same(what):
        for name, a, b in zip(("heads", "records", "decays", "win_pos"), whole.tensors(), other.tensors()):
            assert torch.equal(a, b), (what, name)

    for what, pos in (("any fill", rank % W), ("all due", torch.full_like(rank, W - 1)), ("full and parked", torch.where(rank % 7 == 0, W + 1, rank % (W + 1))), ("the last one", last)):
        whole.win_pos.copy_(pos)
        for a, b in zip(other.tensors(), whole.tensors()):
            a.copy_(b)
        q, k = (x / x.norm(dim=-1, keepdim=True) for x in (normal(batch, heads, 128), normal(batch, heads, 128)))
        alpha = torch.sigmoid(normal(batch, heads, 128) if gate == K else normal(batch, heads))
        tok = [x.to(torch.bfloat16).view(torch.int16).contiguous() for x in (q, k, normal(batch, heads, 128), torch.sigmoid(normal(batch, heads)), alpha)]
        lq.decode_step(shape(batch), whole, *tok, o[0])
        for c, st in zip(cuts, parts):
            lq.decode_step(shape(c.stop - c.start), st, *(x[c] for x in tok), o[1][c])
        assert torch.equal(o[0], o[1]), what
        same(what)
    for force in (False, True):
        whole.win_pos.copy_(rank % (W + 1))
        other.win_pos.copy_(whole.win_pos)
        lq.window_flush(shape(batch), whole, force=force)
        for c, st in zip(cuts, parts):
            lq.window_flush(shape(c.stop - c.start), st, force=force)
        same(f"window_flush, force {force}")
    assert lq.check_device() == 0


@pytest.mark.parametrize("r,bf16,n_iter", [(4, 0, 1), (4, 0, 2), (3, 0, 1), (0, 0, 1), (0, 1, 1)])
def test_states_quantized_by_four_warps_and_by_eight_give_the_same_bits(r, bf16, n_iter):
    """On both sides of the numbers of states where the other number of warps is taken: one, two, three and ten to an SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shape = lambda n: lq.Shape(n, 1, 1, 128, 128, 8, r, n_iter, G, 0 if bf16 else 1, 1, 0, bf16)
    most = 10 * sms + 1
    S = torch.randn((most, 1, 128, 128), generator=torch.Generator("cuda").manual_seed(r), device="cuda")
    want = torch.cat([_quantized(shape(min(100, most - b)), S[b:b + 100]) for b in range(0, most, 100)])
    for n in (k * sms + e for k in (1, 2, 3, 10) for e in (0, 1)):
        assert torch.equal(_quantized(shape(n), S[:n]), want[:n]), n
    assert lq.check_device() == 0


def _quantized(sh, S):
    st = lq.State(sh)
    lq.quantize_state(sh, S, st)
    assert not st.win_pos.any()
    return st.heads
