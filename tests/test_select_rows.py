"""The lane-per-row first stage and the 16-row double-precision stage of the selection at the edges of
their tiles: numbers of candidates around 32, 64 and 128 (odd and even), one block more than the kernels
take, short last tiles, every block size, the non-causal candidates, and rows whose logits lie so far
below the norm bound that single precision gives up.  Bit for bit what double precision everywhere
selects, and the oracle's choice."""
import numpy as np
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_indices

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,dtype,lens,opts", [
    (2, 2, 2, 33 * 32 - 5, 64, 32, 6, "bf16", None, {}),
    (1, 4, 2, 65 * 16, 32, 16, 9, "bf16", (200, 1040), {}),
    (1, 2, 2, 128 * 16, 32, 16, 5, "bf16", None, {}),          # the last number of blocks the kernels take
    (1, 2, 2, 129 * 16 - 15, 32, 16, 5, "bf16", None, {}),     # and the first they do not
    (2, 8, 1, 700, 64, 64, 3, "bf16", (1, 700), {}),           # 512 rows per query block: 8 CTAs, 4 passes
    (3, 2, 2, 500, 64, 32, 4, "fp32", (90, 500), {}),
    (2, 2, 2, 777, 64, 32, 6, "bf16", (100, 777), {"causal": 0}),
    (2, 4, 2, 1030, 32, 64, 5, "bf16", None, {"causal": 0}),
    (2, 4, 2, 900, 64, 32, 5, "bf16", (300, 900), {"cmp": (64, 32)}),
    (2, 2, 2, 450, 32, 32, 4, "bf16", None, {"loose": 1}),
    (2, 4, 2, 530, 64, 32, 6, "bf16", (1, 530), {"per_query": 1, "cmp": (64, 32)}),
    (1, 6, 1, 400, 32, 16, 7, "bf16", None, {"per_query": 1}),  # a group of six heads: two passes of four
    (1, 2, 2, 300, 32, 8, 5, "fp32", (20, 300), {"per_query": 1}),
    (2, 2, 2, 350, 64, 16, 4, "bf16", None, {"per_query": 1, "loose": 1}),
])
def test_certified_selection_at_the_edges(B, H, Hkv, L, D, block, topk, dtype, lens, opts):
    import torch
    from paper_2512_13368_b200 import binding, runner
    w = workloads.make("rows", dtype, B, H, L, D, block, topk, 16, seed=L + H, lengths=lens,
                       kv_heads=Hkv if Hkv != H else 0)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    w.cmp_block, w.cmp_stride = opts.get("cmp", (0, 0))
    if opts.get("loose"):   # long keys and queries with small products: their norms say nothing about the logits
        w.q[..., : D // 2], w.k[..., : D // 2] = 0.0, w.k[..., : D // 2] * 300
        w.q[..., D // 2:], w.k[..., D // 2:] = w.q[..., D // 2:] * 40, w.k[..., D // 2:] * 0.02
        w.q, w.k = workloads.quantize(w.q, dtype), workloads.quantize(w.k, dtype)
    p = runner.DeviceProblem(w)
    got = {}
    for exact in (0, 1):
        binding.blossom_debug_switch(binding.SWITCH_EXACT_SELECT, exact)
        try:
            p.idx.fill_(-7)
            p.select()
            torch.cuda.synchronize()
            got[exact] = p.idx.cpu().numpy().copy()
        finally:
            binding.blossom_debug_switch(binding.SWITCH_EXACT_SELECT, -1)
    assert np.array_equal(got[0], got[1])
    check_indices(w, got[0])
