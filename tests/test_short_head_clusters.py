"""The short backward with a group's heads split over the CTAs of a cluster: every split, heads left over
per CTA, key tiles that are all padding, histories shorter than the sums' place in shared memory, and
both sides of each line of the rule.  Against the oracle; repeated calls give the same bits."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu

CASES = [  # B, H, Hkv, L, D, block, topk, window, lengths, options, CTAs that share a key tile
    (3, 4, 2, 1, 32, 16, 1, 1, None, {}, 2),                                   # one position
    (2, 4, 1, 17, 64, 16, 2, 5, (0, 17), {}, 4),                               # tiles smaller than the sums
    (2, 8, 1, 65, 32, 64, 2, 16, (1, 65), {}, 8),
    (3, 16, 2, 130, 64, 32, 3, 8, (2, 130), {"power_law": 1, "cmp": (64, 32)}, 8),   # two groups
    (3, 16, 1, 130, 64, 32, 3, 8, (2, 130), {}, 8),                            # two heads a CTA
    (2, 6, 1, 143, 32, 16, 3, 20, (20, 143), {"causal": 0, "power_law": 3}, 2),      # three heads a CTA
    (2, 12, 1, 250, 32, 16, 5, 40, (9, 250), {}, 4),                           # three heads a CTA
    (64, 4, 1, 33, 32, 16, 2, 9, (0, 33), {}, 4),                              # the last batch with a CTA a head, D = 32
    (65, 4, 1, 33, 32, 16, 2, 9, (0, 33), {}, 2),                              # two heads a CTA
    (193, 4, 1, 20, 32, 16, 2, 9, None, {}, 1),
    (48, 4, 1, 40, 64, 16, 2, 9, (0, 40), {}, 4),                              # the same at D = 64
    (129, 4, 1, 20, 64, 16, 2, 9, None, {}, 1),
]


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,window,lens,opts,ctas", CASES)
def test_backward_against_the_oracle(B, H, Hkv, L, D, block, topk, window, lens, opts, ctas):
    import torch
    from paper_2512_13368_b200 import binding, runner
    pl = opts.get("power_law", 0)
    w = workloads.make("short", "bf16", B, H, L, D, block, topk, window, seed=L + D, lengths=lens, kv_heads=Hkv,
                       stis_mode=1 if pl else 0, stis_block=pl or 1)
    w.causal = opts.get("causal", 1)
    w.cmp_block, w.cmp_stride = opts.get("cmp", (0, 0))
    p = runner.DeviceProblem(w)
    assert binding.blossom_launch_plan(p.params, binding.PLAN_SHORT_SPLIT, lens is not None) == ctas
    binding.blossom_profile_start(64)
    p.step()
    names = {name for name, _ in binding.blossom_profile_stop(64)}
    assert "bwd_short" in names, names
    print(check_forward_backward(w, p.results()))
    first = {k: getattr(p, k).clone() for k in ("dq", "dk", "dv", "dgate")}
    for k in first:
        getattr(p, k).fill_(float("nan"))
    p.backward()
    for k, t in first.items():
        assert torch.equal(t, getattr(p, k)), k
