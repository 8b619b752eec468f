"""The single-precision kernels at the edges of their tiles: one position, one past a 16-row tile,
more than 64 chunks of 16 positions, grouped heads, padding inside a tile, the power-law mask, no causal
mask, logits too far apart for one softmax reference; few tiles (four warps share one) and many."""
import numpy as np
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,window,lens,opts", [
    (1, 1, 1, 1, 32, 16, 1, 1, None, {}),
    (2, 2, 2, 17, 64, 16, 2, 5, (0, 17), {}),
    (3, 4, 2, 130, 64, 32, 3, 33, (7, 130), {}),
    (2, 6, 1, 200, 32, 16, 4, 8, (1, 200), {"power_law": 1, "cmp": (32, 16)}),
    (2, 2, 1, 143, 32, 64, 2, 20, (20, 143), {"causal": 0, "power_law": 3}),
    (1, 2, 2, 1100, 32, 32, 5, 70, None, {}),        # 69 chunks: two words of the chunk set
    (64, 2, 2, 180, 32, 16, 4, 32, (1, 180), {}),    # a warp per tile
    (33, 2, 2, 257, 64, 64, 3, 40, (30, 257), {"causal": 0}),
    (2, 2, 2, 128, 64, 16, 4, 24, None, {"std": 6.0}),
    (40, 2, 2, 128, 64, 16, 4, 24, None, {"std": 6.0}),
])
def test_forward_and_backward_against_the_oracle(B, H, Hkv, L, D, block, topk, window, lens, opts):
    import torch
    from paper_2512_13368_b200 import runner
    pl = opts.get("power_law", 0)
    w = workloads.make("fp32-tiles", "fp32", B, H, L, D, block, topk, window, seed=L + D, lengths=lens,
                       kv_heads=Hkv if Hkv != H else 0, stis_mode=1 if pl else 0, stis_block=pl or 1)
    w.causal = opts.get("causal", 1)
    w.cmp_block, w.cmp_stride = opts.get("cmp", (0, 0))
    if opts.get("std"):   # logits of hundreds: softmax references that do not cover every row, tame gradients
        w.q = w.q * np.float32(opts["std"] ** 2)
        w.dout = w.dout * np.float32(0.01)
    p = runner.DeviceProblem(w)
    p.step()
    first = {k: getattr(p, k).clone() for k in ("out", "out_lt", "out_st", "lse", "dq", "dk", "dv", "dgate")}
    print(check_forward_backward(w, p.results()))
    p.step()
    for k, t in first.items():
        assert torch.equal(t, getattr(p, k)), k
