"""The work that users of this library have it do, as timed cases.

A serving loop calls ``decode_step`` once per generated token and layer; that call (with the window boundaries of the
sequences that are due) is most of the cases.  The rest is what surrounds it: the same step from host buffers, taking
prefilled dense states into the window representation (``quantize_state``) and reading them back out
(``dequantize_state``).  Shapes, window lengths and distributions are those of the benchmark configurations of this
repository (``synth.config`` and the sweep of ``bench.py``) or generic ones of the same kind.

A state is brought to where a serving loop finds it: dense states after a few dozen tokens, quantized, a window of real
records behind them, and the sequences at window positions that are uniform over [0, W) in no particular order (requests
are admitted when they come, not sorted by age).  A case's token vectors change from pass to pass.

Results are compared exactly: the library takes every sum in a fixed order and states its results bit for bit, and
everything downstream of the 8-bit codes is a step function of those sums.
"""
import math

import torch

from paper_2609_38166_b200 import lq

D = 128
TOKENS = 8             # different tokens a state holds and goes through in turn
WARM = 24              # tokens behind the dense state (the gate forgets faster than that)

# What every case says (a listed or drawn case overrides some of it)
BASE = {"path": "decode", "gate": "gdn", "batch": 256, "heads_v": 32, "heads_qk": 16, "W": 16, "r": 4, "n_iter": 1, "smooth": 1,
        "delta": 1, "rec16": 0, "state_bf16": 0, "outliers": 0, "tokens": 1}


def _case(**kw):
    return {**BASE, **kw}


def listed():
    return [
        # one head of one sequence through a whole window (16 calls): the smallest calls, where launches count
        _case(name="gdn_single_window", batch=1, heads_v=1, heads_qk=1, tokens=16),
        # a small serving batch: a CTA has one head or two, latency counts
        _case(name="gdn_b32", batch=32),
        # the benchmark batch, and the same with the shortest window of the benchmark (a boundary every eight tokens)
        _case(name="gdn_b256"),
        _case(name="gdn_b256_w8", W=8),
        # a large batch with the longest window of the benchmark
        _case(name="gdn_b1024_w32", batch=1024, W=32),
        # per-channel gate with outlier channels; the same gate with the longest window and twice the compensators
        _case(name="kda_b128_outliers", gate="kda", batch=128, heads_qk=32, outliers=1),
        _case(name="kda_b512_w64_r8", gate="kda", batch=512, heads_qk=32, W=64, r=8),
        # an instance without the delta rule at odd sizes, with the fp16 record buffer
        _case(name="gla_ragged_rec16", gate="kda", batch=77, heads_v=12, heads_qk=4, W=13, r=3, delta=0, rec16=1),
        # the per-window BF16 state format
        _case(name="gdn_b256_bf16_state", r=0, smooth=0, state_bf16=1),
        # tokens that arrive in, and outputs that go to, pinned host memory
        _case(name="gdn_b256_host", path="host"),
        # admission of prefilled sequences, and reading states in mid-window back out
        _case(name="gdn_b64_quantize", path="quantize", batch=64),
        _case(name="kda_b64_dequantize", path="dequantize", gate="kda", batch=64, heads_qk=32),
    ]


def draw(rng):
    """One more case of the same ranges."""
    path = rng.choice(("decode",) * 8 + ("host", "quantize", "dequantize"))
    gate = rng.choice(("gdn", "kda"))
    heads_qk = rng.choice((1, 2, 4, 8, 16, 32))
    heads_v = heads_qk * rng.choice((1, 1, 2, 3, 4))
    heads_v = heads_v if heads_v <= 64 else heads_qk
    most = {"decode": 1024, "host": 256, "quantize": 128, "dequantize": 128}[path]
    batch = max(1, round(math.exp(rng.uniform(0.0, math.log(most)))))
    W = rng.choice((8, 16, 16, 32, 64, rng.randint(3, 64)))
    bf16 = rng.random() < 0.12
    case = _case(path=path, gate=gate, batch=batch, heads_v=heads_v, heads_qk=heads_qk, W=W, r=0 if bf16 else rng.choice((2, 3, 4, 4, 4, 6, 8)),
                 n_iter=rng.choice((1, 1, 1, 2)), smooth=0 if bf16 else 1, delta=int(rng.random() < 0.8), rec16=int(rng.random() < 0.3),
                 state_bf16=int(bf16), outliers=int(rng.random() < 0.3))
    top = max(_cost(c) for c in listed())
    while _cost(case) > top:
        case["batch"] = max(1, case["batch"] * 2 // 3)
    return case


def _cost(case):
    """A rough measure of a pass: bytes, with a dense state in fp32 worth of traffic for every window boundary."""
    heads = case["batch"] * case["heads_v"]
    due = heads if case["path"] == "quantize" else heads / case["W"] if case["path"] in ("decode", "host") else 0
    return case["tokens"] * (_bytes(case) + due * (8 * D * D) * (1 + case["r"] / 4) * case["n_iter"])


# ---- inputs ----

def _shape(case):
    return lq.Shape(case["batch"], case["heads_v"], case["heads_qk"], D, D, case["W"], case["r"], case["n_iter"],
                    lq.GATE_DIAG if case["gate"] == "kda" else lq.GATE_SCALAR, case["smooth"], case["delta"], case["rec16"], case["state_bf16"])


class _Tokens:
    """Seeded inputs of decode tokens on the GPU: q, k L2-normalised, v normal, beta a sigmoid, alpha = exp(-softplus) of
    normals; with outliers, 2 % of the key and value channels of a head are eight times as large."""

    def __init__(self, case, seed):
        self.case = case
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed))
        B, H, G = case["batch"], case["heads_v"], case["heads_qk"]
        self.mk = self.mv = None
        if case["outliers"]:
            self.mk, self.mv = (1.0 + 7.0 * (torch.rand((B, h, D), generator=self.gen, device="cuda") < 0.02) for h in (G, H))

    def normal(self, *shape):
        return torch.randn(shape, generator=self.gen, device="cuda")

    def draw(self):
        c = self.case
        B, H, G = c["batch"], c["heads_v"], c["heads_qk"]
        q, k, v = self.normal(B, G, D), self.normal(B, G, D), self.normal(B, H, D)
        if self.mk is not None:
            k, v = k * self.mk, v * self.mv
        q, k = (x / x.norm(dim=-1, keepdim=True) for x in (q, k))
        beta = torch.sigmoid(self.normal(B, H))
        alpha = torch.exp(-torch.nn.functional.softplus(self.normal(B, H, D) if c["gate"] == "kda" else self.normal(B, H)))
        return [x.to(torch.bfloat16).view(torch.int16).contiguous() for x in (q, k, v, beta, alpha)]


def prepare(case, seed):
    sh = _shape(case)
    B, H, W = case["batch"], case["heads_v"], case["W"]
    draws = _Tokens(case, seed)
    o = torch.zeros((case["tokens"], B, H, D), dtype=torch.float32, device="cuda")
    S = torch.zeros((B, H, D, D), dtype=torch.float32, device="cuda")
    for _ in range(WARM):
        lq.ref_decode_step_f32(sh, S, *draws.draw(), o[0])
    st = lq.State(sh)
    s = {"sh": sh, "st": st, "o": o, "i": 0, "path": case["path"]}
    if case["path"] == "quantize":
        s["S"] = S
        return s
    lq.quantize_state(sh, S, st)
    for _ in range(W - 1):                       # a window of records behind every sequence, without a boundary
        lq.decode_step(sh, st, *draws.draw(), o[0])
    order = torch.randperm(B, generator=draws.gen, device="cuda")
    st.win_pos.copy_((order % W).to(torch.int32))        # every sequence where it was after that many of those tokens
    if case["path"] == "dequantize":
        s["S"] = S
        return s
    s["tokens"] = [draws.draw() for _ in range(TOKENS)]
    if case["path"] == "host":
        s["tokens"] = [[x.cpu().pin_memory() for x in tok] for tok in s["tokens"]]
        s["o"] = torch.zeros((B, H, D), dtype=torch.float32).pin_memory()
        s["stage"] = torch.empty((lq.decode_stage_bytes(sh),), dtype=torch.uint8, device="cuda")
    return s


# ---- the pass ----

def run(s):
    sh, st = s["sh"], s["st"]
    state = {"heads": st.heads, "records": st.records, "decays": st.decays, "win_pos": st.win_pos}
    if s["path"] == "quantize":
        lq.quantize_state(sh, s["S"], st)
        return {"heads": st.heads, "win_pos": st.win_pos}
    if s["path"] == "dequantize":
        lq.dequantize_state(sh, st, s["S"])
        return s["S"]
    if s["path"] == "host":
        tok = s["tokens"][s["i"] % TOKENS]
        s["i"] += 1
        lq.decode_step_host_pipelined(sh, st, *tok, s["o"], s["stage"])
        return {"o": s["o"], **state}
    for o in s["o"]:
        tok = s["tokens"][s["i"] % TOKENS]
        s["i"] += 1
        lq.decode_step(sh, st, *tok, o)
    return {"o": s["o"], **state}


# ---- what a pass cannot do without ----

def _bytes(case):
    """Bytes of one token (or one conversion) of the whole batch: every input read once, every output written once."""
    heads = case["batch"] * case["heads_v"]
    W, diag = case["W"], case["gate"] == "kda"
    block = 2 * D * D if case["state_bf16"] else D * D + 8 * D + 4 * D * case["r"]
    record = (2 if case["rec16"] else 4) * (3 if diag else 2) * D + (0 if diag else 4)
    if case["path"] == "quantize":
        return heads * (4 * D * D + block)
    held = heads * (block + (W - 1) / 2 * record)            # window positions are uniform over [0, W)
    if case["path"] == "dequantize":
        return held + heads * 4 * D * D
    token = 2 * 2 * case["batch"] * case["heads_qk"] * D + heads * (2 * D + 2 + (2 * D if diag else 2))
    return held + token + heads * (4 * D + record) + heads / W * block


def work(case):
    heads = case["batch"] * case["heads_v"]
    W, r = case["W"], case["r"]
    rebuild = 2 * D * D * (r + 2)                            # codes to values, compensators, decay
    quantize = 2 * D * D * (3 * r * case["n_iter"] + 4)      # fit (two products per round), removal, smoothing, scales, codes
    if case["path"] == "quantize":
        return {"bytes": _bytes(case), "flops": heads * quantize}
    if case["path"] == "dequantize":
        return {"bytes": _bytes(case), "flops": heads * (rebuild + 2 * D * D * (W - 1) / 2)}
    readout = 2 * (2 * D * D + 4 * D * (r + (W - 1) / 2))
    boundary = (rebuild + 2 * D * D * W + (0 if case["state_bf16"] else quantize)) / W
    return {"bytes": case["tokens"] * _bytes(case), "flops": case["tokens"] * heads * (readout + boundary)}


def tolerance(case):
    return "exact"
