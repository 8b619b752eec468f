"""The short-history kernels (one launch per direction) at the edges of their tiles and of their rule:
one position, one past a 16-row tile or a block, ragged last blocks, padding that starts inside a
tile, both head dimensions, grouped heads, logits too far apart for one softmax reference, and the
largest sizes of either side of the rule.  Against the oracle; skipped selection and exact ties too."""
import numpy as np
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward, check_indices

pytestmark = pytest.mark.gpu

CASES = [  # B, H, Hkv, L, D, block, topk, window, lengths, options
    (1, 1, 1, 1, 32, 16, 1, 1, None, {}),
    (2, 2, 2, 17, 64, 16, 2, 5, (0, 17), {}),
    (3, 2, 2, 65, 32, 64, 2, 16, (1, 65), {}),
    (3, 4, 2, 129, 64, 32, 3, 33, (7, 129), {}),
    (2, 6, 2, 250, 32, 16, 5, 40, (9, 250), {"power_law": 1}),
    (2, 8, 2, 200, 64, 16, 4, 8, (1, 200), {"power_law": 1, "cmp": (32, 16)}),
    (2, 2, 1, 143, 32, 16, 3, 20, (20, 143), {"causal": 0}),
    (2, 2, 2, 143, 64, 32, 3, 20, (20, 143), {"causal": 0, "power_law": 3}),
    (9, 4, 4, 400, 32, 16, 6, 50, (30, 400), {}),       # the largest training length of the rule
    (33, 2, 2, 300, 64, 32, 4, 64, (1, 300), {}),       # short forward, general backward
    (56, 2, 2, 300, 64, 32, 4, 64, (1, 300), {}),       # (the row above is still within the short backward's rule, this is not)
    (2, 2, 2, 128, 64, 16, 4, 24, None, {"std": 9.0}),  # logits of several hundred
    (2, 2, 2, 96, 32, 16, 3, 10, None, {"ties": 1}),
]


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,window,lens,opts", CASES)
def test_forward_and_backward_against_the_oracle(B, H, Hkv, L, D, block, topk, window, lens, opts):
    import torch
    from paper_2512_13368_b200 import binding, runner
    pl = opts.get("power_law", 0)
    w = workloads.make("short", "bf16", B, H, L, D, block, topk, window, seed=L + D, lengths=lens,
                       std=opts.get("std", 1.0), kv_heads=Hkv if Hkv != H else 0, stis_mode=1 if pl else 0,
                       stis_block=pl or 1)
    w.causal = opts.get("causal", 1)
    w.cmp_block, w.cmp_stride = opts.get("cmp", (0, 0))
    if opts.get("ties"):
        w.k[:] = w.k[:, :, :1, :]
    p = runner.DeviceProblem(w)
    n0 = binding.blossom_launch_count()
    p.forward()
    assert binding.blossom_launch_count() - n0 == 1
    p.backward()
    # (with equal keys dq vanishes analytically: a relative bar says nothing there)
    print(check_forward_backward(w, p.results(), backward=not opts.get("ties")))
    first = {k: getattr(p, k).clone() for k in ("out", "dq", "dk", "dv", "dgate")}
    p.backward()                      # on the same workspace again, then as a call of its own
    p.backward(reuse_tile_lists=False)
    for k, t in first.items():
        assert torch.equal(t, getattr(p, k)), k
    out = p.out.clone()
    p.out.fill_(float("nan"))
    p.forward(idx_is_input=True)      # the same indices given
    assert torch.equal(out, p.out)


@pytest.mark.parametrize("L,H,D", [(257, 1, 64), (512, 2, 32), (512, 4, 64)])
def test_forward_only_up_to_the_largest_length(L, H, D):
    from paper_2512_13368_b200 import binding, runner
    w = workloads.make("short-serve", "bf16", 3, H, L, D, 32, 6, 40, seed=L, lengths=(1, L))
    p = runner.DeviceProblem(w, training=False)
    n0 = binding.blossom_launch_count()
    p.forward()
    assert binding.blossom_launch_count() - n0 == 1
    res = p.results()
    check_indices(w, res["idx"])
    print(check_forward_backward(w, res, backward=False))
