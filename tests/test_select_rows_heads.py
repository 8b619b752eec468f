"""The selection per query position with a group's heads over the warps that share rows: groups that take one round of
two or four heads, several rounds, and none; both sides of the line on the number of tiles; lengths that end inside
a warp's rows; overlapping compression blocks.  Index rows against the oracle."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_indices

pytestmark = pytest.mark.gpu

CASES = [  # B, H, Hkv, L, D, block, topk, lengths, compression block and stride
    (3, 4, 1, 300, 64, 32, 4, (1, 300), 0, 0),      # four heads at once
    (2, 8, 1, 257, 32, 16, 5, (40, 257), 0, 0),     # two rounds of four
    (2, 6, 1, 200, 32, 16, 4, None, 0, 0),          # three rounds of two
    (2, 3, 1, 200, 64, 32, 3, (33, 200), 0, 0),     # a head after the other
    (2, 4, 2, 700, 64, 64, 4, (100, 700), 128, 64),  # blocks larger than a CTA's rows, Eq. 11
    (2, 8, 2, 330, 32, 32, 3, (5, 330), 64, 32),
    (224, 4, 2, 97, 32, 16, 3, (1, 97), 32, 16),    # 448 tiles: the last with heads side by side
    (225, 4, 2, 97, 32, 16, 3, (1, 97), 32, 16),    # 450
]


@pytest.mark.parametrize("B,H,Hkv,L,D,block,topk,lens,cmp_block,cmp_stride", CASES)
def test_heads_side_by_side(B, H, Hkv, L, D, block, topk, lens, cmp_block, cmp_stride):
    from paper_2512_13368_b200 import runner
    w = workloads.make("heads", "bf16", B, H, L, D, block, topk, 8, seed=L + H, lengths=lens, kv_heads=Hkv)
    w.per_query, w.cmp_block, w.cmp_stride = 1, cmp_block, cmp_stride
    p = runner.DeviceProblem(w)
    p.forward()
    check_indices(w, p.results()["idx"])
