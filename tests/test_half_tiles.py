"""Pairs of half tiles of 32 rows in the tensor-core kernels: odd numbers of halves in a list and in either phase (an
odd one is paired with the half behind the last), lists of one half, a last half that the sequence does not fill, halves
that only the window or only a selection needs, padding that ends inside a half.  Against the oracle."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu

CASES = [  # B, H, Hkv, L, D, block, topk, window, lengths, options
    (2, 2, 2, 321, 64, 32, 3, 1, None, {}),                         # eleven halves, one key in the last
    (6, 2, 2, 352, 32, 32, 4, 40, (1, 352), {}),                    # padding that ends in every place of a half
    (3, 2, 2, 415, 64, 16, 4, 33, (20, 415), {}),                   # two blocks a half
    (3, 2, 2, 480, 64, 64, 3, 20, (30, 480), {}),                   # one block over two halves
    (2, 4, 2, 353, 64, 32, 4, 8, (100, 353), {"power_law": 1}),     # packed heads; links to single halves
    (3, 2, 2, 360, 64, 32, 2, 25, (33, 360), {"causal": 0}),
    (2, 4, 2, 350, 32, 32, 3, 8, (90, 350), {"per_query": 1, "power_law": 1}),
    (2, 2, 2, 333, 64, 64, 3, 30, None, {"per_query": 1}),
]


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,window,lens,opts", CASES)
def test_odd_halves(B, H, Hkv, L, D, block, topk, window, lens, opts):
    from paper_2512_13368_b200 import runner
    w = workloads.make("halves", "bf16", B, H, L, D, block, topk, window, seed=L + block, lengths=lens,
                       kv_heads=Hkv if Hkv != H else 0, stis_mode=opts.get("power_law", 0), stis_block=1)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    p = runner.DeviceProblem(w)
    p.step()
    print(check_forward_backward(w, p.results()))
