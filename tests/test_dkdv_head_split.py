"""dK and dV of grouped heads on either side of the rule that splits a group's heads over clusters: one, two and
four CTAs a key tile.  Against the oracle."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Hkv,L,D", [
    (80, 4, 1, 450, 64),    # 320 key tiles: the last with 2 CTAs each
    (81, 4, 1, 450, 64),    # one
    (40, 2, 1, 450, 64),    # 160, two heads: the last with 2
    (41, 2, 1, 450, 64),    # one
    (48, 4, 1, 450, 32),    # 192: 2, and not 4
    (24, 4, 1, 450, 32),    # 96: 4, the last
])
def test_either_side_of_the_rule(B, H, Hkv, L, D):
    from paper_2512_13368_b200 import runner
    w = workloads.make("split", "bf16", B, H, L, D, 32, 4, 20, seed=B, lengths=(1, L), kv_heads=Hkv)
    p = runner.DeviceProblem(w)
    p.step()
    print(check_forward_backward(w, p.results()))
