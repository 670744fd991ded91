"""GPU: which heads a window boundary takes.  The kernels find the due sequences by looking over all window positions; the
sizes here are where that can go wrong: one sequence, more sequences than one load of every thread covers (256) and than one
trip does (2048), more due heads per CTA than one list holds (32), in one trip and in several, windows in random order, all due at once, none due."""
import numpy as np
import pytest
import torch

from oracle.lq_oracle import State as OState
from paper_2609_38166_b200 import lq, synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("state_bf16", [0, 1])
@pytest.mark.parametrize("batch,heads_v,heads_qk,W,order", [(1, 1, 1, 4, "last"), (5, 3, 3, 5, "all"), (300, 3, 1, 4, "random"),
                                                            (257, 2, 2, 3, "none"), (301, 32, 16, 2, "all"),
                                                            (2049, 1, 1, 3, "last"), (2500, 2, 1, 4, "random"), (4750, 2, 1, 2, "all")])
def test_boundaries_of_windows_in_any_order(oracle, batch, heads_v, heads_qk, W, order, state_bf16):
    kw = dict(r=0, smooth=0, state_bf16=1) if state_bf16 else dict(r=2)
    wl = synth.Workload("due", batch, heads_v, heads_qk, W=W, seed=800 + batch, **kw)
    osh, lsh = gu.shapes(wl)
    ost = OState(osh)
    oracle.quantize_state(osh, synth.dense_states(wl, 3), ost)
    rng = np.random.default_rng(batch)
    ost.win_pos[:] = {"last": np.where(np.arange(batch) == batch - 1, W - 1, np.arange(batch) % W), "all": np.full(batch, W - 1),
                      "random": rng.integers(0, W, batch), "none": np.zeros(batch)}[order]
    ost.buf_k[...] = rng.standard_normal(ost.buf_k.shape).astype(np.float32) * 0.1
    ost.buf_u[...] = rng.standard_normal(ost.buf_u.shape).astype(np.float32)
    ost.buf_a[...] = rng.uniform(0.2, 1.0, ost.buf_a.shape).astype(np.float32)
    st = gu.state_to_dev(ost, lsh)
    o = torch.empty((batch, heads_v, 128), dtype=torch.float32, device="cuda")
    for step in range(2):
        tok = synth.token_inputs(wl, step)
        want = oracle.decode_step(osh, ost, **tok)
        td = gu.tok_dev(tok)
        lq.decode_step(lsh, st, td["q"], td["k"], td["v"], td["beta"], td["alpha"], o)
        assert np.array_equal(gu.host(o), want), f"o of step {step}"
        gu.assert_state_parity(st, ost, wl.r, f"state after step {step}")
    lq.window_flush(lsh, st, force=True)            # every window that holds records, whatever its fill
    oracle.window_flush(osh, ost, force=True)
    gu.assert_state_parity(st, ost, wl.r, "forced flush")
    assert st.win_pos.tolist() == [0] * batch and lq.check_device() == 0


@pytest.mark.parametrize("r", [3, 12])
@pytest.mark.parametrize("shift", [0, 4])
def test_dense_states_at_any_16_byte_boundary(oracle, shift, r):
    """Dense states come by bulk copies (up to eight compensators) or are loaded, and stored, 32 bytes at a time where their
    base allows it; a base that is only 16-byte aligned (`shift` floats into an allocation) takes the other branch."""
    wl = synth.Workload("al", 3, 2, 1, W=5, r=r, seed=830)
    osh, lsh = gu.shapes(wl)
    S0 = synth.dense_states(wl, 3)
    ost = OState(osh)
    oracle.quantize_state(osh, S0, ost)
    room = torch.zeros(S0.size + 8, dtype=torch.float32, device="cuda")
    S = room[shift:shift + S0.size].view(S0.shape)
    S.copy_(gu.dev(S0))
    st = lq.State(lsh)
    lq.quantize_state(lsh, S, st)
    gu.assert_state_parity(st, ost, wl.r, "quantize")
    S.zero_()
    lq.dequantize_state(lsh, st, S)
    assert np.array_equal(gu.host(S), oracle.dequantize_state(osh, ost))
    assert not room[:shift].any() and not room[shift + S0.size:].any()


@pytest.mark.parametrize("gate", [synth.GATE_SCALAR, synth.GATE_DIAG])
def test_many_windows_that_come_in_full_among_drawn_heads(oracle, gate):
    """More than three heads per resident CTA, most of them of sequences that enter with a full window and get no token: the
    CTAs draw many such heads in a row.  Their outputs stay, the boundary takes all of them, the others step as usual."""
    wl = synth.Workload("fullw", 90, 32, 16, W=4, r=2, gate=gate, seed=840)
    osh, lsh = gu.shapes(wl)
    ost = OState(osh)
    oracle.quantize_state(osh, synth.dense_states(wl, 3), ost)
    rng = np.random.default_rng(3)
    pos = np.where(rng.random(wl.batch) < 0.8, wl.W, rng.integers(0, wl.W, wl.batch)).astype(np.int32)
    pos[:4] = 1
    ost.win_pos[:] = pos
    ost.buf_k[...] = rng.standard_normal(ost.buf_k.shape).astype(np.float32) * 0.1
    ost.buf_u[...] = rng.standard_normal(ost.buf_u.shape).astype(np.float32)
    ost.buf_a[...] = rng.uniform(0.2, 1.0, ost.buf_a.shape).astype(np.float32)
    st = gu.state_to_dev(ost, lsh)
    o = torch.full((wl.batch, wl.heads_v, 128), 7.0, dtype=torch.float32, device="cuda")
    tok = synth.token_inputs(wl, 0)
    td = gu.tok_dev(tok)
    lq.decode_step(lsh, st, td["q"], td["k"], td["v"], td["beta"], td["alpha"], o)
    torch.cuda.synchronize()
    assert lq.check_device() == 0 and not st.work.any()
    full = torch.from_numpy(pos == wl.W)
    assert torch.all(o.cpu()[full] == 7.0) and not torch.any(o.cpu()[~full] == 7.0)
    assert st.win_pos.tolist() == [0 if p >= wl.W - 1 else int(p) + 1 for p in pos]
    few = np.concatenate([np.flatnonzero(pos == wl.W)[:3], np.arange(3)])      # a few sequences of either kind, by the oracle
    sub = wl.with_(batch=1)
    osub, _ = gu.shapes(sub)
    for b in few:
        one = OState(osub)
        for name in ("codes", "col_scale", "row_smooth", "comp_k", "comp_u", "buf_k", "buf_u", "buf_a", "win_pos"):
            getattr(one, name)[...] = getattr(ost, name)[b:b + 1]
        if pos[b] == wl.W:
            oracle.window_flush(osub, one, force=False)
        else:
            want = oracle.decode_step(osub, one, **{k: np.ascontiguousarray(v[b:b + 1]) for k, v in tok.items()})
            assert np.array_equal(gu.host(o)[b:b + 1], want)
        assert np.array_equal(gu.gpu_codes(st)[b:b + 1], one.codes) and np.array_equal(gu.host(st.col_scale)[b:b + 1], one.col_scale)


@pytest.mark.parametrize("state_bf16", [0, 1])
@pytest.mark.parametrize("gate", [synth.GATE_SCALAR, synth.GATE_DIAG])
def test_full_windows_between_heads_with_a_token(oracle, gate, state_bf16):
    """Several heads per resident CTA, taken in turn (no scratch words), with sequences that enter with a full window in
    between: such a head meets at no barrier, and the two warps hand kt^T q from one to the other through two words in turn.
    Sixteen compensators make the reader of that word late."""
    kw = dict(r=0, smooth=0, state_bf16=1) if state_bf16 else dict(r=16)
    wl = synth.Workload("between", 60, 48, 16, W=3, gate=gate, seed=845, **kw)
    osh, lsh = gu.shapes(wl)
    ost = OState(osh)
    oracle.quantize_state(osh, synth.dense_states(wl, 3), ost)
    rng = np.random.default_rng(5)
    ost.buf_k[...] = rng.standard_normal(ost.buf_k.shape).astype(np.float32) * 0.1
    ost.buf_u[...] = rng.standard_normal(ost.buf_u.shape).astype(np.float32)
    ost.buf_a[...] = rng.uniform(0.2, 1.0, ost.buf_a.shape).astype(np.float32)
    pieces = ["buf_k", "buf_u", "buf_a", "win_pos"] + (["S0"] if state_bf16 else ["codes", "col_scale", "row_smooth", "comp_k", "comp_u"])
    for pattern in range(4):
        full = np.arange(wl.batch) % 2 == pattern if pattern < 2 else rng.random(wl.batch) < 0.4
        ost.win_pos[:] = np.where(full, wl.W, rng.integers(0, wl.W, wl.batch))
        st = gu.state_to_dev(ost, lsh, work=False)
        assert lq.step_launches(lsh, st) == 2
        o = torch.full((wl.batch, wl.heads_v, 128), 7.0, dtype=torch.float32, device="cuda")
        tok = synth.token_inputs(wl, pattern)
        td = gu.tok_dev(tok)
        lq.decode_step(lsh, st, td["q"], td["k"], td["v"], td["beta"], td["alpha"], o)
        some = wl.with_(batch=int((~full).sum()))
        osub, _ = gu.shapes(some)
        sub = OState(osub)
        for name in pieces:
            getattr(sub, name)[...] = getattr(ost, name)[~full]
        want = oracle.decode_step(osub, sub, **{k: np.ascontiguousarray(v[~full]) for k, v in tok.items()})
        got = gu.host(o)
        assert np.array_equal(got[~full], want) and (got[full] == 7.0).all(), pattern
        assert np.array_equal(gu.host_f32(st.buf_u)[~full], sub.buf_u), pattern
    assert lq.check_device() == 0


@pytest.mark.parametrize("batch,launches", [(40, 2), (20, 1)])
def test_parked_sequences_hold_up_nobody(oracle, batch, launches):
    """Sequences at a position above W (the caller's mark for "no request here": 2^31 - 1, -1, 65535, W + 1; the first sequence
    among them) get no token, keep their position and their rows of the output, and the windows of the others go on."""
    wl = synth.Workload("parked", batch, 4, 2, W=3, r=2, seed=850 + batch)
    osh, lsh = gu.shapes(wl)
    ost = OState(osh)
    oracle.quantize_state(osh, synth.dense_states(wl, 3), ost)
    marks = {0: 2 ** 31 - 1, 3: -1, 5: 65535, batch - 1: wl.W + 1}
    parked = np.isin(np.arange(batch), list(marks))
    st = gu.state_to_dev(ost, lsh)
    assert lq.step_launches(lsh, st) == launches
    for b, mark in marks.items():
        st.win_pos[b] = mark
    some = wl.with_(batch=int((~parked).sum()))
    osub, _ = gu.shapes(some)
    sub = OState(osub)
    for name in ("codes", "col_scale", "row_smooth", "comp_k", "comp_u", "win_pos"):
        getattr(sub, name)[...] = getattr(ost, name)[~parked]
    o = torch.full((batch, 4, 128), 7.0, dtype=torch.float32, device="cuda")
    for step in range(3 * wl.W + 1):
        tok = synth.token_inputs(wl, step)
        td = gu.tok_dev(tok)
        lq.decode_step(lsh, st, td["q"], td["k"], td["v"], td["beta"], td["alpha"], o)
        want = oracle.decode_step(osub, sub, **{k: np.ascontiguousarray(v[~parked]) for k, v in tok.items()})
        got = gu.host(o)
        assert np.array_equal(got[~parked], want) and (got[parked] == 7.0).all(), step
        assert st.win_pos.cpu().numpy()[~parked].tolist() == sub.win_pos.tolist(), step
        assert {b: int(st.win_pos[b]) for b in marks} == marks, step
    lq.window_flush(lsh, st)                 # nothing is full
    assert np.array_equal(gu.gpu_codes(st)[~parked], sub.codes)
    lq.window_flush(lsh, st, force=True)     # the others' windows, whatever becomes of the parked ones
    oracle.window_flush(osub, sub, force=True)
    assert np.array_equal(gu.gpu_codes(st)[~parked], sub.codes) and not st.win_pos.cpu().numpy()[~parked].any()
    assert lq.check_device() == 0
