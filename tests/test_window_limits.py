"""Windows and mask blocks of the whole history and beyond, up to the largest int ("no limit"): the same bits
from every kernel family, and the oracle's."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu

INT_MAX = 2 ** 31 - 1
CASES = [  # dtype, H, Hkv, L, D, block, lengths, options
    ("bf16", 2, 2, 90, 32, 16, (5, 90), {}),
    ("bf16", 2, 2, 90, 64, 16, None, {"causal": 0}),
    ("bf16", 4, 2, 130, 32, 32, (40, 130), {"power_law": 1}),
    ("bf16", 2, 2, 600, 64, 64, (100, 600), {}),
    ("bf16", 2, 2, 530, 32, 32, None, {"causal": 0}),
    ("bf16", 4, 2, 600, 64, 32, None, {"power_law": 1}),
    ("bf16", 2, 2, 600, 32, 32, None, {"power_law": 1, "causal": 0}),
    ("fp32", 2, 2, 100, 32, 16, (9, 100), {}),
    ("fp32", 2, 2, 100, 64, 16, None, {"causal": 0, "power_law": 1}),
    ("fp32", 2, 2, 70, 32, 8, (9, 70), {}),
    ("fp32", 2, 2, 70, 32, 8, None, {"causal": 0, "power_law": 1}),
]


@pytest.mark.parametrize("dtype,H,Hkv,L,D,block,lens,opts,what", [c + ("window",) for c in CASES] +
                         [c + ("mask_block",) for c in CASES if c[-1].get("power_law")])
def test_limits_past_the_sequence(dtype, H, Hkv, L, D, block, lens, opts, what):
    import torch
    from paper_2512_13368_b200 import runner
    first = None
    for x in (L, L + 1, 2 * L, INT_MAX - 16, INT_MAX):
        w = workloads.make("limits", dtype, 2, H, L, D, block, 3, x if what == "window" else 9, seed=L, lengths=lens,
                           kv_heads=Hkv if Hkv != H else 0, stis_mode=opts.get("power_law", 0),
                           stis_block=x if what == "mask_block" else 1)
        w.causal = opts.get("causal", 1)
        p = runner.DeviceProblem(w)
        p.step()
        torch.cuda.synchronize()
        got = {k: getattr(p, k).clone() for k in ("idx", "out", "out_lt", "out_st", "lse", "dq", "dk", "dv", "dgate")}
        if first is None:
            first = got
            check_forward_backward(w, p.results())
        for k, t in got.items():
            assert torch.equal(t, first[k]), (x, k)
