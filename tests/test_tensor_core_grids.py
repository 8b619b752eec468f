"""The persistent forward and the grids behind it at the edges of their rules: tiles one fewer, as many and
more than the CTAs that fit, tiles without any row to do, head-packed tiles, lists too long for a second
buffer, dK/dV with a group's heads split over two and four CTAs, and the two passes of the input-dependent
gate.  Against the oracle."""
import numpy as np
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward, check_indices

pytestmark = pytest.mark.gpu

CASES = [  # B, H, Hkv, L, D, block, topk, window, lengths, options
    (59, 1, 1, 577, 64, 64, 3, 40, (1, 577), {}),               # 295 tiles of 128 rows, most short
    (37, 2, 2, 512, 64, 32, 4, 70, (0, 512), {}),               # 296: one for every CTA
    (33, 3, 3, 370, 64, 32, 4, 20, (0, 370), {}),               # 297
    (100, 2, 2, 431, 32, 16, 5, 33, (30, 431), {}),             # 800, blocks of 16
    (20, 8, 4, 520, 64, 64, 3, 30, (1, 520), {}),               # 720 packed tiles; two heads of a group over two CTAs
    (3, 8, 2, 700, 64, 32, 5, 8, (90, 700), {"power_law": 1}),  # four heads of a group over a cluster of four
    (1, 2, 2, 3400, 64, 64, 6, 50, None, {"per_query": 1}),     # lists of 10 KB: one buffer
    (2, 4, 2, 900, 64, 64, 4, 60, (300, 900), {"gate": 1}),     # both passes with a cluster of two
    (5, 2, 2, 777, 32, 32, 4, 60, (1, 777), {"gate": 1, "causal": 0}),
]


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,window,lens,opts", CASES)
def test_forward_and_backward_against_the_oracle(B, H, Hkv, L, D, block, topk, window, lens, opts):
    from paper_2512_13368_b200 import runner
    w = workloads.make("grids", "bf16", B, H, L, D, block, topk, window, seed=L + B, lengths=lens,
                       kv_heads=Hkv if Hkv != H else 0, stis_mode=opts.get("power_law", 0), stis_block=1)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    if opts.get("gate"):
        w.gate_mode = 1
        w.gate = (0.3 * np.random.default_rng(L).standard_normal((H, 2 * D + 1))).astype(np.float32)
    p = runner.DeviceProblem(w)
    p.forward()
    p.backward()
    res = p.results()
    check_indices(w, res["idx"])
    print(check_forward_backward(w, res))
