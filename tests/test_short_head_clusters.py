"""The short backward with a group's heads split over the CTAs of a cluster: every split, heads left over
per CTA, key tiles that are all padding, histories shorter than the sums' place in shared memory, and
both sides of each line of the rule.  Against the oracle; repeated calls give the same bits."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu

CASES = [  # B, H, Hkv, L, D, block, topk, window, lengths, options
    (3, 4, 2, 1, 32, 16, 1, 1, None, {}),                                   # 2 CTAs, one position
    (2, 4, 1, 17, 64, 16, 2, 5, (0, 17), {}),                               # 4 CTAs, tiles smaller than the sums
    (2, 8, 1, 65, 32, 64, 2, 16, (1, 65), {}),                              # 8 CTAs
    (3, 16, 2, 130, 64, 32, 3, 8, (2, 130), {"power_law": 1, "cmp": (64, 32)}),   # 8 CTAs with two heads each
    (2, 6, 1, 143, 32, 16, 3, 20, (20, 143), {"causal": 0, "power_law": 3}),      # 2 CTAs with three heads each
    (2, 12, 1, 250, 32, 16, 5, 40, (9, 250), {}),                           # 4 CTAs with three heads each
    (64, 4, 1, 33, 32, 16, 2, 9, (0, 33), {}),                              # the last batch with 4 CTAs, D = 32
    (65, 4, 1, 33, 32, 16, 2, 9, (0, 33), {}),                              # 2 CTAs with two heads each
    (193, 4, 1, 20, 32, 16, 2, 9, None, {}),                                # none
    (48, 4, 1, 40, 64, 16, 2, 9, (0, 40), {}),                              # the same at D = 64
    (129, 4, 1, 20, 64, 16, 2, 9, None, {}),
]


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,window,lens,opts", CASES)
def test_backward_against_the_oracle(B, H, Hkv, L, D, block, topk, window, lens, opts):
    import torch
    from paper_2512_13368_b200 import runner
    pl = opts.get("power_law", 0)
    w = workloads.make("short", "bf16", B, H, L, D, block, topk, window, seed=L + D, lengths=lens, kv_heads=Hkv,
                       stis_mode=1 if pl else 0, stis_block=pl or 1)
    w.causal = opts.get("causal", 1)
    w.cmp_block, w.cmp_stride = opts.get("cmp", (0, 0))
    p = runner.DeviceProblem(w)
    p.step()
    print(check_forward_backward(w, p.results()))
    first = {k: getattr(p, k).clone() for k in ("dq", "dk", "dv", "dgate")}
    for k in first:
        getattr(p, k).fill_(float("nan"))
    p.backward()
    for k, t in first.items():
        assert torch.equal(t, getattr(p, k)), k
