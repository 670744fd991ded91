"""GPU: a step of more heads than SMs in one launch (tokens and boundaries side by side) against the same step in two.  A state
without the scratch words takes two launches always, so each case steps two copies of a state, one with and one without the words, and
every array has to end with the same bits.  The sizes are where the one launch can go wrong: one head more than the decode kernel has
CTAs (six to an SM; up to there both copies take two launches), several due heads for a CTA, all heads due, none, windows that come in full, parked sequences, three and four slots to an SM, the longest
list of sequences, few sequences of many heads and the reverse, and the largest numbers of heads that are taken this way."""
import numpy as np
import pytest
import torch

from oracle.lq_oracle import State as OState
from paper_2609_38166_b200 import lq, synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

G, K = synth.GATE_SCALAR, synth.GATE_DIAG


def _tokens(sh, gen):
    B, H, Q = sh.batch, sh.heads_v, sh.heads_qk
    n = lambda *s: torch.randn(s, generator=gen, device="cuda")
    q, k = (x / x.norm(dim=-1, keepdim=True) for x in (n(B, Q, 128), n(B, Q, 128)))
    alpha = torch.exp(-torch.nn.functional.softplus(n(B, H, 128) if sh.gate == K else n(B, H)))
    return [x.to(torch.bfloat16).view(torch.int16).contiguous() for x in (q, k, n(B, H, 128), torch.sigmoid(n(B, H)), alpha)]


@pytest.mark.parametrize("gate,batch,heads_v,heads_qk,W,r,n_iter,plain", [
    (G, 149, 1, 1, 16, 4, 1, 0), (K, 149, 1, 1, 9, 4, 1, 0),         # one head more than SMs (of 148)
    (G, 32, 16, 4, 8, 4, 1, 0), (K, 40, 10, 5, 7, 3, 1, 0),          # a pair has a head or two
    (G, 64, 32, 16, 16, 8, 1, 0), (K, 61, 37, 1, 16, 6, 2, 0),       # drawn heads; more than four compensators, several rounds
    (G, 50, 7, 7, 4, 0, 1, 0), (K, 50, 7, 1, 4, 0, 1, 1), (G, 29, 11, 11, 5, 1, 3, 1),
    (G, 200, 1, 1, 2, 2, 1, 0), (K, 33, 9, 3, 3, 4, 1, 0),           # short windows
    (G, 20, 32, 16, 40, 4, 1, 0), (K, 40, 16, 16, 28, 5, 1, 0),      # three slots to an SM
    (G, 96, 64, 16, 32, 4, 1, 0), (G, 256, 32, 16, 24, 2, 1, 0),     # long windows, more due heads than SMs
    (G, 2048, 1, 1, 14, 4, 1, 0), (K, 1025, 2, 2, 16, 4, 1, 0), (G, 3, 64, 1, 16, 4, 1, 0),
    (G, 888, 1, 1, 16, 4, 1, 0), (G, 889, 1, 1, 16, 4, 1, 0), (K, 889, 1, 1, 9, 4, 1, 0),        # the last of two launches and the first of one (148 SMs)
    (G, 64, 16, 4, 8, 4, 1, 0), (K, 100, 10, 5, 7, 3, 1, 0), (G, 14, 64, 1, 16, 2, 1, 0), (G, 90, 11, 11, 8, 1, 1, 1), (K, 64, 32, 32, 16, 8, 1, 0),
    (G, 128, 7, 7, 8, 0, 1, 0), (K, 150, 7, 1, 8, 0, 1, 1), (G, 128, 32, 16, 32, 0, 1, 0),
    (G, 222, 8, 8, 12, 4, 2, 0), (G, 170, 11, 11, 14, 1, 3, 1), (G, 128, 32, 16, 32, 4, 2, 0), (K, 64, 32, 32, 16, 8, 2, 0),       # several rounds: from twelve to an SM on,
    (G, 111, 8, 8, 4, 4, 2, 0), (G, 112, 8, 8, 9, 4, 2, 0), (K, 112, 8, 8, 10, 8, 2, 0), (K, 100, 10, 5, 7, 8, 3, 0),              # or where two SMs of three have a due head
    (G, 40, 32, 16, 40, 4, 1, 0), (K, 60, 16, 16, 28, 5, 1, 0), (K, 128, 32, 32, 32, 4, 1, 0),   # three slots, the last with drawn heads
    (G, 120, 32, 16, 24, 8, 1, 0), (K, 80, 32, 32, 20, 2, 1, 0)])                                # drawn heads with r > 4; diagonal gate, four slots
def test_one_launch_of_many_heads_and_two_give_the_same_bits(gate, batch, heads_v, heads_qk, W, r, n_iter, plain):
    sh = lq.Shape(batch, heads_v, heads_qk, 128, 128, W, r, n_iter, gate, 0 if plain else 1, 0 if plain else 1, 0, 0)
    gen = torch.Generator("cuda").manual_seed(batch * W + r)
    one, two = lq.State(sh), lq.State(sh, work=False)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    heads = batch * heads_v
    few = heads <= 6 * sms or (n_iter > 1 and heads <= 12 * sms and 3 * heads <= 2 * sms * W)
    assert lq.step_launches(sh, one) == (2 if few else 1) and lq.step_launches(sh, two) == 2
    lq.quantize_state(sh, torch.randn((batch, heads_v, 128, 128), generator=gen, device="cuda"), one)
    one.records.copy_(0.2 * torch.randn(one.records.shape, generator=gen, device="cuda"))
    one.decays.copy_(torch.rand(one.decays.shape, generator=gen, device="cuda") * 0.8 + 0.2)
    if gate == K:
        one.records[..., 256:] = torch.rand(one.records[..., 256:].shape, generator=gen, device="cuda") * 0.8 + 0.2
    for name in ("heads", "records", "decays"):
        getattr(two, name).copy_(getattr(one, name))
    o = [torch.full((batch, heads_v, 128), 7.0, dtype=torch.float32, device="cuda") for _ in range(2)]
    rank = torch.randperm(batch, generator=gen, device="cuda").to(torch.int32)
    patterns = [rank % W, torch.full_like(rank, W - 1), torch.where(rank % 3 == 0, W, rank % W), rank % (W + 1), torch.full_like(rank, W),
                torch.where(rank % 5 == 1, 2 ** 31 - 1, torch.where(rank % 5 == 2, W + 1, rank % W)), torch.zeros_like(rank),
                torch.where(rank == 0, W - 1, 0)]
    for i, pos in enumerate(patterns):
        for st in (one, two):
            st.win_pos.copy_(pos)
        for _ in range(2):
            tok = _tokens(sh, gen)
            lq.decode_step(sh, one, *tok, o[0])
            lq.decode_step(sh, two, *tok, o[1])
        assert torch.equal(o[0], o[1]), f"o, pattern {i}"
        for name in ("win_pos", "heads", "records", "decays"):
            assert torch.equal(getattr(one, name), getattr(two, name)), f"{name}, pattern {i}"
        assert not one.work.any(), f"scratch words, pattern {i}"
    assert lq.check_device() == 0


@pytest.mark.parametrize("gate,batch,heads", [(G, 128, 8), (K, 112, 9)])
def test_one_launch_of_many_heads_against_the_oracle_and_in_a_graph(oracle, gate, batch, heads):
    """A window and a half of steps, windows of every fill: called one by one against the oracle, and captured once and replayed."""
    wl = synth.Workload("merged", batch, heads, heads, W=8, r=4, gate=gate, seed=1300 + gate)
    osh, sh = gu.shapes(wl)
    ost = OState(osh)
    oracle.quantize_state(osh, synth.dense_states(wl, 2), ost)
    ost.win_pos[:] = np.random.default_rng(4).permutation(batch) % wl.W
    ost.buf_a[...] = 1.0
    states = [gu.state_to_dev(ost, sh) for _ in range(2)]
    assert lq.step_launches(sh, states[0]) == 1
    toks = [synth.token_inputs(wl, t) for t in range(12)]
    tds = [[gu.tok_dev(t)[x] for x in ("q", "k", "v", "beta", "alpha")] for t in toks]
    outs = [torch.zeros((12, batch, heads, 128), dtype=torch.float32, device="cuda") for _ in range(2)]
    for t, tok in enumerate(toks):
        lq.decode_step(sh, states[0], *tds[t], outs[0][t])
        assert np.array_equal(gu.host(outs[0][t]), oracle.decode_step(osh, ost, **tok)), t
    gu.assert_state_parity(states[0], ost, wl.r, "after the steps")
    g, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=stream):
        for t in range(12):
            lq.decode_step(sh, states[1], *tds[t], outs[1][t], stream)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1])
    for a, b in zip(states[0].tensors(), states[1].tensors()):
        assert torch.equal(a, b)
    assert not states[1].work.any() and lq.check_device() == 0
