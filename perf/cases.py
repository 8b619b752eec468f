"""Workloads a user of the library runs, as plain cases that can be prepared, run and timed.

Two users stand behind them.  A model author calls ``autograd.blossom_attention`` inside a
PyTorch program (training steps, and evaluation under ``no_grad``).  A serving or training runtime
with buffers of its own calls the C ABI through ``binding`` and keeps outputs and workspace from
one call to the next.  The sizes are those of the repository's configurations (``workloads.py``,
``bench.py`` and its flags, ``layer_step.py``), of the paper's own history lengths (50 and 200
positions), and their neighbourhood: from one request of one user to whole training batches of
long histories, left-padded batches and lengths that are no multiple of anything.

A case is a dict: ``entry`` ("autograd" or "abi"), ``train`` (forward + backward, else forward
only), ``dtype``, the sizes B, H, Hkv, L, D, the selection (block, topk, window), ``min_len``
(0: every sequence is full; else lengths are drawn from [min_len, L]), ``std`` of q, k, v and
whether their rows have norms of their own (``row_scales``), ``grad_layout`` (how the upstream
gradient arrives: "bhld" dense like q, or "blhd", the transposed view that a projection after the
attention hands back), and the options of the path: ``power_law``, ``cmp_block`` / ``cmp_stride``,
``per_query``, ``causal``, ``input_gate``, ``rope_theta``.
"""
import math

import torch

from paper_2512_13368_b200 import binding
from paper_2512_13368_b200.autograd import blossom_attention

_BASE = dict(entry="autograd", train=True, dtype="bf16", B=1, H=2, Hkv=2, L=200, D=32, block=16, topk=4,
             window=32, min_len=0, std=1.0, row_scales=False, grad_layout="bhld", power_law=False,
             cmp_block=0, cmp_stride=0, per_query=False, causal=True, input_gate=False, rope_theta=0.0)


def _case(**kw):
    c = dict(_BASE, **kw)
    if "Hkv" not in kw:
        c["Hkv"] = c["H"]
    return c


def listed():
    return [
        # one request of one user with a short history, evaluated inside a PyTorch program
        _case(name="serve-one", train=False, B=1, H=2, L=50, D=32),
        # a serving batch of short, left-padded histories; the runtime keeps its buffers
        _case(name="serve-batch-padded", entry="abi", train=False, B=64, H=2, L=200, D=32, min_len=5, std=0.5),
        # one user with a very long history (the headline configuration's shape at batch 1)
        _case(name="serve-long", train=False, B=1, H=8, L=4096, D=64, block=64, topk=16, window=256),
        # training on short padded histories (configuration 2)
        _case(name="train-short-padded", B=256, H=2, L=200, D=32, min_len=5, std=0.5),
        # the same kind of batch for a model trained in single precision
        _case(name="train-short-fp32", dtype="fp32", B=128, H=2, L=200, D=32, min_len=5, std=0.5),
        # the paper's default options at the paper's history length: 8 heads on 2 key/value heads,
        # overlapping compression blocks, power-law mask
        _case(name="train-paper-options", B=128, H=8, Hkv=2, L=200, D=32, window=8, power_law=True,
              cmp_block=32, cmp_stride=16, min_len=20),
        # mid-length training (configuration 3: per-row norms spread out)
        _case(name="train-mid", B=128, H=4, L=1024, D=64, block=32, topk=8, window=64, row_scales=True),
        # the attention of the layer case (configuration 5); the gradient arrives as the transposed
        # view that the projection behind the attention hands back
        _case(name="train-layer", B=128, H=2, L=1024, D=32, block=32, topk=8, window=64, grad_layout="blhd"),
        # the headline configuration (4) with the caller's own buffers, as bench.py runs it
        _case(name="train-long", entry="abi", B=16, H=8, L=4096, D=64, block=64, topk=16, window=256),
        # the paper's options with its selection per query position
        _case(name="train-paper-per-query", B=8, H=8, Hkv=2, L=1500, D=64, block=32, topk=8, window=8,
              power_law=True, cmp_block=64, cmp_stride=32, per_query=True, min_len=200),
        # a bidirectional encoder (no causal mask) on ragged lengths
        _case(name="train-bidirectional", B=16, H=4, L=777, D=64, block=32, topk=6, window=70, causal=False,
              min_len=100),
        # input-dependent gate and rotary positions inside the library
        _case(name="train-gate-rope", B=16, H=4, L=900, D=64, block=32, topk=5, window=70, input_gate=True,
              rope_theta=10000.0, min_len=200),
    ]


# ---- drawn cases: the families above over their ranges ---------------------------------------
def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["serve", "serve", "short", "short", "fp32", "paper", "paper-per-query", "mid", "mid",
                       "long", "bidirectional", "gate-rope"])
    c = dict(_BASE)
    c["D"] = rng.choice([32, 64])
    c["H"] = c["Hkv"] = rng.choice([1, 2, 4, 8])
    c["std"] = rng.choice([0.5, 1.0])
    c["grad_layout"] = rng.choice(["bhld", "bhld", "blhd"])
    if kind == "serve":
        c["train"], c["L"] = False, _log_int(rng, 20, 4096)
    elif kind == "short":
        c["L"] = _log_int(rng, 40, 400)
    elif kind == "fp32":
        c["dtype"], c["L"] = "fp32", _log_int(rng, 40, 400)
    elif kind == "paper":
        c["L"] = _log_int(rng, 50, 1200)
    elif kind == "paper-per-query":
        c["L"] = _log_int(rng, 50, 1500)
    elif kind == "mid":
        c["L"], c["row_scales"] = _log_int(rng, 300, 1500), rng.random() < 0.5
    elif kind == "long":
        c["L"] = _log_int(rng, 1500, 4096)
    else:
        c["L"] = _log_int(rng, 100, 1500)
    L = c["L"]
    c["block"] = 16 if L <= 300 else 32 if L <= 1500 else 64
    if 300 < L <= 1500 and kind in ("mid", "serve") and rng.random() < 0.3:
        c["block"] = 64
    c["topk"] = rng.randint(3, 5) if L <= 300 else rng.randint(5, 9) if L <= 1500 else rng.randint(10, 16)
    c["window"] = rng.randint(8, 48) if L <= 300 else rng.randint(32, 128) if L <= 1500 else rng.randint(64, 256)
    if kind.startswith("paper"):
        c["H"], c["Hkv"] = 8, rng.choice([2, 2, 4])
        c["power_law"], c["window"] = True, rng.choice([8, 16])
        c["cmp_block"], c["cmp_stride"] = 2 * c["block"], c["block"]
        c["per_query"] = kind == "paper-per-query"
    elif kind == "bidirectional":
        c["causal"] = False
    elif kind == "gate-rope":
        c["input_gate"] = True
        c["rope_theta"] = rng.choice([0.0, 10000.0])
    if rng.random() < 0.5:
        c["min_len"] = rng.randint(1, max(1, L // 2))
    if rng.random() < 0.3 and not c["input_gate"]:
        c["entry"] = "abi"
        c["grad_layout"] = "bhld"
    # the batch: small ones for serving, otherwise up to what fits a tenth of the largest listed case
    # (the options without a certified single-precision selection, and single precision, cost more a row)
    per_seq = work(dict(c, B=1))
    weight = {"fp32": 24.0, "paper-per-query": 4.0, "bidirectional": 3.0, "gate-rope": 2.0}.get(kind, 1.0)
    largest = work(listed()[8])
    room = min(largest["flops"] / (per_seq["flops"] * weight), largest["bytes"] / (per_seq["bytes"] * weight))
    cap = max(1, min(1024, int(room * (0.9 if kind == "long" else 0.3))))
    c["B"] = _log_int(rng, 1, min(cap, 64)) if kind == "serve" else _log_int(rng, max(1, cap // 16), cap)
    return c


# ---- inputs ------------------------------------------------------------------------------------
class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = c = case
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(int(seed) % (1 << 62))
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    B, H, Hkv, L, D = c["B"], c["H"], c["Hkv"], c["L"], c["D"]

    def normal(shape, std=1.0):
        return torch.randn(shape, generator=g, device=dev) * std

    def rows(h):
        x = normal((B, h, L, D), c["std"])
        if c["row_scales"]:
            x *= torch.rand((B, h, L, 1), generator=g, device=dev) * 1.5 + 0.5
        return x.to(dt)

    s.q, s.k, s.v = rows(H), rows(Hkv), rows(Hkv)
    s.gate = normal((H, 2 * D + 1), 0.2) if c["input_gate"] else normal((H, 2))
    s.lens = None
    if c["min_len"]:
        s.lens = torch.randint(c["min_len"], L + 1, (B,), generator=g, device=dev, dtype=torch.int32)
    if c["train"]:
        if c["grad_layout"] == "blhd":
            s.dout = normal((B, L, H, D)).to(dt).transpose(1, 2)
        else:
            s.dout = normal((B, H, L, D)).to(dt)
    if c["entry"] == "abi":
        s.params = binding.make_params(
            B, H, L, D, c["block"], c["topk"], c["window"], c["dtype"], kv_heads=Hkv,
            causal=int(c["causal"]), select_mode=int(c["per_query"]), stis_mode=int(c["power_law"]),
            cmp_block=c["cmp_block"], cmp_stride=c["cmp_stride"], gate_mode=int(c["input_gate"]),
            rope_theta=c["rope_theta"])
        s.params_bwd = binding.blossom_params.from_buffer_copy(s.params)
        s.params_bwd.reuse_tile_lists = 1
        index_rows = L if c["per_query"] else -(-L // c["block"])
        s.idx = torch.empty((B, Hkv, index_rows, c["topk"]), dtype=torch.int32, device=dev)
        s.out = torch.empty_like(s.q)
        s.out_lt = s.out_st = s.lse = None
        if c["train"]:
            s.out_lt, s.out_st = torch.empty_like(s.q), torch.empty_like(s.q)
            s.lse = torch.empty((2, B, H, L), dtype=torch.float32, device=dev)
            s.dq, s.dk, s.dv = torch.empty_like(s.q), torch.empty_like(s.k), torch.empty_like(s.v)
            s.dgate = torch.empty_like(s.gate)
        s.workspace = torch.empty(binding.blossom_workspace_bytes(s.params), dtype=torch.uint8, device=dev)
    elif c["train"]:
        for t in (s.q, s.k, s.v, s.gate):
            t.requires_grad_(True)
    return s


# ---- one pass ----------------------------------------------------------------------------------
def run(state):
    s, c = state, state.case
    if c["entry"] == "abi":
        binding.blossom_attn_fwd(s.params, s.q, s.k, s.v, s.gate, s.lens, s.idx, 0, s.out, s.out_lt, s.out_st,
                                 s.lse, s.workspace)
        if not c["train"]:
            return {"out": s.out, "idx": s.idx}
        binding.blossom_attn_bwd(s.params_bwd, s.q, s.k, s.v, s.gate, s.lens, s.idx, s.out_lt, s.out_st, s.lse,
                                 s.dout, s.dq, s.dk, s.dv, s.dgate, s.workspace)
        return {"out": s.out, "idx": s.idx, "dq": s.dq, "dk": s.dk, "dv": s.dv, "dgate": s.dgate}

    def attention():
        return blossom_attention(
            s.q, s.k, s.v, s.gate, c["block"], c["topk"], c["window"], seq_lens=s.lens, return_indices=True,
            short_term="power-law" if c["power_law"] else "window", cmp_block=c["cmp_block"],
            cmp_stride=c["cmp_stride"], select_per_query=c["per_query"],
            input_dependent_gate=c["input_gate"], causal=c["causal"], rope_theta=c["rope_theta"])

    if not c["train"]:
        with torch.no_grad():
            out, idx = attention()
        return {"out": out, "idx": idx}
    out, idx = attention()
    dq, dk, dv, dgate = torch.autograd.grad(out, (s.q, s.k, s.v, s.gate), s.dout)
    return {"out": out, "idx": idx, "dq": dq, "dk": dk, "dv": dv, "dgate": dgate}


# ---- what a pass cannot do without ---------------------------------------------------------------
def _pairs(c, n):
    """(query, key) pairs of one head for a sequence of n valid positions: long-term branch, short-term
    branch, and (query, scored block) pairs of the selection."""
    L, bk, k, w = c["L"], c["block"], c["topk"], c["window"]
    pad0 = L - n
    b0 = pad0 // bk
    lt = st = sc = 0
    stride, length = c["cmp_stride"] or bk, c["cmp_block"] or bk
    for b in range(b0, -(-L // bk)):
        lo, hi = max(b * bk, pad0), min((b + 1) * bk, L)
        m = hi - lo
        if c["causal"]:
            cand = b - b0
            lt += m * min(k - 1, cand) * bk + m * (m + 1) // 2
            sc += m * max(0, (b * bk - pad0 - length) // stride + 1) if cand > k - 1 else 0
        else:
            cand = -(-L // bk) - b0 - 1
            lt += m * (min(k - 1, cand) * bk + m)
            sc += m * cand if cand > k - 1 else 0
    one_side = sum(min(t, w - 1) for t in range(min(n, w))) + max(0, n - w) * (w - 1)
    st = n + (one_side if c["causal"] else 2 * one_side)
    if c["power_law"]:  # keys at power-of-two distances outside the window
        d = 1
        while d < n:
            if d >= w:
                st += (n - d) * (1 if c["causal"] else 2)
            d *= 2
    return lt, st, sc


def work(case):
    c = case
    B, H, Hkv, L, D = c["B"], c["H"], c["Hkv"], c["L"], c["D"]
    esz = 2 if c["dtype"] == "bf16" else 4
    lo = c["min_len"] or L
    lens = [L] if lo == L else [lo + (L - lo) * (2 * i + 1) // 16 for i in range(8)]  # quantiles of the drawn lengths
    lt = st = sc = 0.0
    for n in lens:
        a, b, d = _pairs(c, n)
        lt, st, sc = lt + a / len(lens), st + b / len(lens), sc + d / len(lens)
    gemms = 7 if c["train"] else 2  # forward S, PV; backward S, dP, dV, dK, dQ
    flops = B * H * 2.0 * D * (gemms * (lt + st) + sc)
    share = sum(lens) / len(lens) / L  # padded rows are not read; output rows are all written
    q_in, kv_in, q_out, kv_out = B * H * L * D * share, 2 * B * Hkv * L * D * share, B * H * L * D, 2 * B * Hkv * L * D
    elems = q_in + kv_in + q_out
    if c["train"]:
        elems += q_in + q_out + kv_out  # the upstream gradient; dq, dk, dv
    index_rows = L if c["per_query"] else -(-L // c["block"])
    return {"bytes": elems * esz + 4.0 * B * Hkv * index_rows * c["topk"], "flops": flops}


def tolerance(case):
    # bf16 storage: probabilities and their gradients are rounded to bf16 (2^-9) between the products;
    # single precision: sums of a few hundred fp32 terms and fp32 exponentials.  Block indices are the
    # choice a double-precision evaluation makes: the same whole numbers.
    return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 2e-5}
