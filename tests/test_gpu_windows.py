"""GPU: windows of every fill, for the shapes whose records reach the decode kernel in segments (two of 8 fp32 or 12 fp16 rows
at a time) and the neighbours that take them at once; remainders of every size, both gates, both state formats."""
import numpy as np
import pytest
import torch

from oracle.lq_oracle import State as OState
from paper_2609_38166_b200 import lq, synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

G, K = synth.GATE_SCALAR, synth.GATE_DIAG


@pytest.mark.parametrize("gate,W,rec16,state_bf16", [(G, 32, 0, 0), (G, 40, 0, 0), (G, 64, 1, 0), (K, 24, 0, 0), (K, 32, 0, 0), (K, 63, 0, 0),
                                                     (K, 64, 1, 0), (G, 24, 0, 1), (G, 64, 1, 1), (K, 32, 1, 1), (K, 64, 0, 1), (G, 2, 0, 1)])
def test_every_fill_of_a_window(oracle, gate, W, rec16, state_bf16):
    kw = dict(r=0, smooth=0, state_bf16=1) if state_bf16 else dict(r=3)
    wl = synth.Workload("fill", W, 8, 4, W=W, gate=gate, rec16=rec16, seed=850 + W, **kw)
    osh, lsh = gu.shapes(wl)
    ost = OState(osh)
    oracle.quantize_state(osh, synth.dense_states(wl, 3), ost)
    rng = np.random.default_rng(W)
    ost.win_pos[:] = rng.permutation(W)
    half = lambda a: a.astype(np.float16).astype(np.float32)        # (values that either record format holds)
    ost.buf_k[...] = half(rng.standard_normal(ost.buf_k.shape) * 0.1)
    ost.buf_u[...] = half(rng.standard_normal(ost.buf_u.shape))
    ost.buf_a[...] = half(rng.uniform(0.9, 1.0, ost.buf_a.shape))
    st = gu.state_to_dev(ost, lsh)
    assert lq.step_launches(lsh, st) == (1 if W == 2 else 2)
    o = torch.empty((W, 8, 128), dtype=torch.float32, device="cuda")
    for step in range(2):
        tok = synth.token_inputs(wl, step)
        want = oracle.decode_step(osh, ost, **tok)
        td = gu.tok_dev(tok)
        lq.decode_step(lsh, st, td["q"], td["k"], td["v"], td["beta"], td["alpha"], o)
        assert np.array_equal(gu.host(o), want), f"o of step {step}"
        gu.assert_state_parity(st, ost, wl.r, f"state after step {step}")
    assert lq.check_device() == 0


@pytest.mark.parametrize("gate,W,rec16", [(G, 3, 0), (G, 9, 1), (G, 24, 0), (K, 9, 0)])
def test_bf16_state_several_heads_per_cta(oracle, gate, W, rec16):
    """Per-window BF16, three and more heads per resident CTA: the records of a CTA's next head are asked for while this one's
    state is multiplied, so every lane must be through with the rows before; every fill of a window, a boundary included."""
    wl = synth.Workload("bfmany", 60, 48, 16, W=W, gate=gate, rec16=rec16, r=0, smooth=0, state_bf16=1, seed=880 + W)
    osh, lsh = gu.shapes(wl)
    ost = OState(osh)
    oracle.quantize_state(osh, synth.dense_states(wl, 3), ost)
    rng = np.random.default_rng(W)
    ost.win_pos[:] = rng.permutation(wl.batch) % W
    half = lambda a: a.astype(np.float16).astype(np.float32)
    ost.buf_k[...] = half(rng.standard_normal(ost.buf_k.shape, dtype=np.float32) * 0.1)
    ost.buf_u[...] = half(rng.standard_normal(ost.buf_u.shape, dtype=np.float32))
    ost.buf_a[...] = half(rng.uniform(0.5, 1.0, ost.buf_a.shape))
    st = gu.state_to_dev(ost, lsh)
    assert lq.step_launches(lsh, st) == 2
    o = torch.empty((wl.batch, wl.heads_v, 128), dtype=torch.float32, device="cuda")
    for step in range(2):
        tok = synth.token_inputs(wl, step)
        want = oracle.decode_step(osh, ost, **tok)
        td = gu.tok_dev(tok)
        lq.decode_step(lsh, st, td["q"], td["k"], td["v"], td["beta"], td["alpha"], o)
        assert np.array_equal(gu.host(o), want), f"o of step {step}"
        gu.assert_state_parity(st, ost, wl.r, f"state after step {step}")
    assert lq.check_device() == 0
