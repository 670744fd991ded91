"""GPU: a step of few heads is one launch (a CTA per head takes the token and the boundary), a step of more heads is two.  The
same sequences stepped both ways have to end with the same bits, over two windows in every state of filling."""
import pytest
import torch

from paper_2609_38166_b200 import lq, synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

G, K = synth.GATE_SCALAR, synth.GATE_DIAG
HEADS = 4


def _shape(batch, W, r, gate, rec16, bf16, n_iter, plain):
    """`plain`: without the delta rule and without residual smoothing"""
    return lq.Shape(batch, HEADS, 2, 128, 128, W, r, n_iter, gate, 0 if bf16 or plain else 1, 0 if plain else 1, rec16, bf16)


@pytest.mark.parametrize("gate,W,r,rec16,bf16,n_iter,plain", [
    (G, 16, 4, 0, 0, 1, 0), (G, 1, 2, 0, 0, 1, 0), (G, 2, 0, 0, 0, 1, 0), (G, 5, 8, 1, 0, 2, 0), (G, 64, 3, 1, 0, 1, 0), (G, 40, 16, 0, 0, 1, 0),
    (K, 16, 4, 0, 0, 1, 0), (K, 12, 4, 1, 0, 1, 0), (G, 11, 4, 1, 0, 2, 0), (K, 6, 8, 0, 0, 1, 0), (K, 7, 0, 1, 0, 1, 0), (K, 33, 5, 0, 0, 1, 0), (K, 64, 16, 0, 0, 2, 0), (K, 13, 9, 1, 0, 1, 0),
    (G, 16, 0, 0, 1, 1, 0), (G, 9, 0, 1, 1, 1, 0), (K, 64, 0, 0, 1, 1, 0), (K, 3, 0, 1, 1, 1, 0),
    (G, 7, 4, 0, 0, 1, 1), (K, 5, 3, 0, 0, 1, 1), (G, 6, 8, 1, 0, 1, 1), (K, 9, 0, 1, 1, 1, 1)])
def test_one_launch_and_two_give_the_same_bits(gate, W, r, rec16, bf16, n_iter, plain):
    few = torch.cuda.get_device_properties(0).multi_processor_count // HEADS        # the most sequences of one launch
    B = 2 * few
    whole, part = _shape(B, W, r, gate, rec16, bf16, n_iter, plain), _shape(few, W, r, gate, rec16, bf16, n_iter, plain)
    kw = dict(r=0, smooth=0, state_bf16=1) if bf16 else dict(r=r)
    wl = synth.Workload("one", B, HEADS, 2, W=W, gate=gate, rec16=rec16, seed=900 + W, **kw)
    S = torch.randn((B, HEADS, 128, 128), generator=torch.Generator("cuda").manual_seed(W), device="cuda")
    st = lq.State(whole)
    assert lq.step_launches(whole, st) == 2 and lq.step_launches(part, lq.State(part)) == 1
    lq.quantize_state(whole, S, st)
    cuts = [slice(0, few), slice(few, B)]
    parts = []
    for cut in cuts:
        parts.append(lq.State(part))
        parts[-1].heads.copy_(st.heads[cut])
    o, o_part = (torch.zeros((n, HEADS, 128), dtype=torch.float32, device="cuda") for n in (B, few))
    spread = torch.arange(B, dtype=torch.int32, device="cuda")
    for step in range(2 * W + 2):
        if step == W:                        # windows of every fill from here on, some of them full (no token, the boundary only)
            for s, at in ((st, spread), (parts[0], spread[cuts[0]]), (parts[1], spread[cuts[1]])):
                s.win_pos.copy_(at % (W + 1))
        tok = gu.tok_dev(synth.token_inputs(wl, step))
        args = [tok[x] for x in ("q", "k", "v", "beta", "alpha")]
        lq.decode_step(whole, st, *args, o)
        for cut, s in zip(cuts, parts):
            o_part.copy_(o[cut])             # (a sequence without a token leaves its rows as they are)
            o_part[:, :, 0] += 1.0
            before = o_part.clone()
            token = (s.win_pos < W)[:, None, None]
            lq.decode_step(part, s, *(a[cut].contiguous() for a in args), o_part)
            assert torch.equal(o_part, torch.where(token, o[cut], before)), f"o of step {step}"
            for name in ("win_pos", "heads", "records", "decays"):
                assert torch.equal(getattr(s, name), getattr(st, name)[cut]), f"{name} after step {step}"
    assert lq.check_device() == 0
