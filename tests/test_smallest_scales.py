"""Logit scales down to the denormals, which single-precision arithmetic here flushes to zero: the softmaxes are
uniform over what a query may see, and what it may not see still counts nothing.  Against the oracle."""
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,L,D,opts", [
    ("bf16", 450, 64, {}),
    ("bf16", 450, 32, {"kv_heads": 2}),
    ("bf16", 450, 64, {"causal": 0}),
    ("bf16", 450, 64, {"per_query": 1}),
    ("bf16", 450, 32, {"stis_mode": 1}),
    ("bf16", 40, 32, {}),
    ("fp32", 150, 64, {}),
])
@pytest.mark.parametrize("scale", [1e-45, 1e-38, 1.2e-38])
def test_uniform_weights(dtype, L, D, opts, scale):
    from paper_2512_13368_b200 import runner
    w = workloads.make("small-scale", dtype, 2, 4, L, D, 32, 4, 20, seed=L, lengths=(L // 3, L),
                       kv_heads=opts.get("kv_heads", 0), stis_mode=opts.get("stis_mode", 0), stis_block=1)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    p = runner.DeviceProblem(w, sm_scale=scale)
    p.step()
    print(check_forward_backward(w, p.results(), sm_scale=scale))
