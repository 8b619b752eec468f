"""Pairs of half tiles in lists of several rounds (a warp lists 64 halves a round), against the oracle; and the same bits from
repeated steps where most pairs are two separate copies, with the outputs poisoned in between."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu

CASES = [  # B, H, Hkv, L, D, block, topk, window, lengths, options
    (1, 2, 2, 2337, 64, 32, 9, 70, None, {}),                              # 74 halves, one row in the last
    (2, 2, 2, 2210, 32, 16, 12, 40, (700, 2210), {}),                      # two blocks a half
    (1, 4, 2, 2400, 64, 32, 8, 8, (2001, 2400), {"power_law": 1}),         # packed heads
    (1, 2, 2, 2150, 64, 32, 6, 90, (2100, 2150), {"causal": 0}),
    (1, 4, 2, 2190, 32, 32, 5, 16, (2150, 2190), {"per_query": 1}),
]


def make(B, H, Hkv, L, D, block, topk, window, lens, opts):
    w = workloads.make("halves", "bf16", B, H, L, D, block, topk, window, seed=L + block, lengths=lens,
                       kv_heads=Hkv if Hkv != H else 0, stis_mode=opts.get("power_law", 0), stis_block=1)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    return w


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,window,lens,opts", CASES)
def test_many_halves(B, H, Hkv, L, D, block, topk, window, lens, opts):
    from paper_2512_13368_b200 import runner
    w = make(B, H, Hkv, L, D, block, topk, window, lens, opts)
    p = runner.DeviceProblem(w)
    p.step()
    print(check_forward_backward(w, p.results()))


@pytest.mark.parametrize("Hkv,D,opts", [(4, 64, {}), (4, 32, {}), (2, 64, {"power_law": 1}), (4, 64, {"causal": 0})])
def test_repeated_steps_with_separate_halves(Hkv, D, opts):
    import torch
    from paper_2512_13368_b200 import runner
    p = runner.DeviceProblem(make(4, 4, Hkv, 2048, D, 32, 8, 100, (700, 2048), opts))
    p.step()
    keys = ("idx", "out", "out_lt", "out_st", "lse", "dq", "dk", "dv", "dgate")
    first = {k: getattr(p, k).clone() for k in keys}
    for it in range(30):
        for k in keys:
            getattr(p, k).view(torch.uint8).fill_(0xFF)
        p.step()
        for k in keys:
            assert torch.equal(first[k].view(torch.uint8), getattr(p, k).view(torch.uint8)), (it, k)
