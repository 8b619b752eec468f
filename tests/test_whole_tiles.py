"""Blocks of 64 in the tensor-core kernels: lists of whole tiles (two adjacent halves).  One tile, a last tile of which the
sequence fills one half or a single row, more tiles than a warp has lanes, padding that ends inside a half, odd numbers of
tiles that only one of a CTA's 64-row halves needs, every mask and option.  Against the oracle."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu

CASES = [  # B, H, Hkv, L, D, topk, window, lengths, options
    (2, 2, 2, 401, 64, 2, 20, None, {}),                        # one row in the last tile
    (4, 2, 2, 416, 32, 4, 64, (1, 416), {}),                    # half a tile at the end, padding that ends in every place
    (1, 2, 2, 2500, 64, 16, 200, None, {}),                     # two rounds of 32 tiles
    (2, 4, 2, 2105, 64, 9, 8, (500, 2105), {"power_law": 1}),   # packed heads, links to single tiles
    (2, 2, 2, 2300, 32, 5, 150, (64, 2300), {"causal": 0}),
    (2, 4, 1, 2200, 64, 6, 30, (900, 2200), {"per_query": 1}),
]


@pytest.mark.parametrize("B,H,Hkv,L,D,topk,window,lens,opts", CASES)
def test_whole_tiles(B, H, Hkv, L, D, topk, window, lens, opts):
    from paper_2512_13368_b200 import runner
    w = workloads.make("whole", "bf16", B, H, L, D, 64, topk, window, seed=L + topk, lengths=lens,
                       kv_heads=Hkv if Hkv != H else 0, stis_mode=opts.get("power_law", 0), stis_block=1)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    p = runner.DeviceProblem(w)
    p.step()
    print(check_forward_backward(w, p.results()))
