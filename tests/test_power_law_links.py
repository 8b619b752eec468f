"""Single links at power-of-two distances in the tensor-core kernels, on both sides without the causal mask:
lengths about the multiples of the 64-column tiles and of the distances where a tile holds one link, two or
none.  Against the oracle."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Hkv,L,D,block,window,causal,per_query,lens", [
    (2, 2, 2, 65, 64, 16, 3, 1, 1, (64, 65)),
    (2, 4, 2, 130, 32, 32, 8, 1, 1, (96, 130)),
    (2, 2, 2, 300, 64, 32, 1, 0, 0, (257, 300)),
    (1, 4, 2, 577, 32, 64, 8, 0, 0, None),
    (1, 2, 1, 1100, 64, 32, 8, 1, 1, None),
    (1, 2, 2, 1090, 64, 32, 40, 0, 0, (1000, 1090)),
])
def test_single_links(B, H, Hkv, L, D, block, window, causal, per_query, lens):
    from paper_2512_13368_b200 import binding, runner
    w = workloads.make("links", "bf16", B, H, L, D, block, 3, window, seed=L, lengths=lens,
                       kv_heads=Hkv if Hkv != H else 0, stis_mode=1, stis_block=1)
    w.causal, w.per_query = causal, per_query
    p = runner.DeviceProblem(w)
    binding.blossom_profile_start(64)
    p.step()
    names = {name for name, _ in binding.blossom_profile_stop(64)}
    assert {"fwd_tc", "bwd_dq_tc", "bwd_dkdv_tc"} <= names, names
    print(check_forward_backward(w, p.results()))
