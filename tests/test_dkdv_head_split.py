"""dK and dV of grouped heads on either side of the rule that splits a group's heads over clusters: one, two and
four CTAs a key tile, with and without lengths and in every form of the kernel.  Against the oracle."""
import numpy as np
import pytest

from paper_2512_13368_b200 import binding, build, workloads
from parity_util import check_forward_backward


@pytest.mark.parametrize("heads,lengths,batches", [
    (2, False, {1: 2, 42: 2, 43: 1}), (2, True, {1: 2, 57: 2, 58: 1}),
    (4, False, {1: 4, 21: 4, 22: 2, 54: 2, 55: 1}), (4, True, {28: 4, 29: 2, 89: 2, 90: 1}),
    (6, False, {1: 2, 66: 2, 67: 1}), (8, False, {27: 4, 28: 2, 78: 2, 79: 1}), (8, True, {44: 4, 45: 2, 153: 2, 154: 1}),
    (1, False, {1: 1}), (3, True, {1: 1}),
])
def test_the_lines(heads, lengths, batches):
    """CTAs that share a key tile of L 450 (four tiles a sequence), one key/value head."""
    build.build()
    for B, want in batches.items():
        p = binding.make_params(B, heads, 450, 64, 32, 4, 20, "bf16", kv_heads=1)
        assert binding.blossom_launch_plan(p, binding.PLAN_DKDV_SPLIT, lengths) == want, B
    fp32 = binding.make_params(1, heads, 450, 64, 32, 4, 20, "fp32", kv_heads=1)
    assert binding.blossom_launch_plan(fp32, binding.PLAN_DKDV_SPLIT, lengths) == 0
    with pytest.raises(binding.BlossomError):
        binding.blossom_launch_plan(fp32, 3, lengths)


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,Hkv,L,D,lens,opts,ctas", [
    (28, 4, 1, 450, 64, (1, 450), {}, 4),           # the last batch with 4
    (29, 4, 1, 450, 64, (1, 450), {}, 2),
    (90, 4, 1, 450, 64, (1, 450), {}, 1),
    (42, 2, 1, 450, 64, None, {}, 2),               # the last with 2
    (43, 2, 1, 450, 64, None, {}, 1),
    (21, 4, 1, 450, 32, None, {}, 4),
    (22, 4, 1, 450, 32, None, {}, 2),
    (3, 8, 2, 450, 64, (1, 450), {"per_query": 1}, 4),
    (40, 4, 2, 450, 32, None, {"per_query": 1}, 1),
    (20, 4, 2, 450, 32, (1, 450), {"per_query": 1}, 2),
    (2, 8, 2, 450, 32, (1, 450), {"causal": 0}, 4),
    (9, 12, 2, 450, 64, None, {"causal": 0}, 2),
    (2, 4, 1, 450, 64, (1, 450), {"gate": 1}, 4),   # two passes, the second adds to the first's
    (5, 6, 1, 450, 32, (1, 450), {"gate": 1}, 2),
    (2, 8, 1, 450, 64, None, {"gate": 1, "causal": 0}, 4),
])
def test_either_side_of_the_rule(B, H, Hkv, L, D, lens, opts, ctas):
    from paper_2512_13368_b200 import runner
    w = workloads.make("split", "bf16", B, H, L, D, 32, 4, 20, seed=B, lengths=lens, kv_heads=Hkv)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    if opts.get("gate"):
        w.gate_mode = 1
        w.gate = (0.3 * np.random.default_rng(L).standard_normal((H, 2 * D + 1))).astype(np.float32)
    p = runner.DeviceProblem(w)
    assert binding.blossom_launch_plan(p.params, binding.PLAN_DKDV_SPLIT, lens is not None) == ctas
    binding.blossom_profile_start(64)
    p.step()
    names = {name for name, _ in binding.blossom_profile_stop(64)}
    assert "bwd_dkdv_tc" in names, names
    print(check_forward_backward(w, p.results()))
