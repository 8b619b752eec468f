"""The single-precision certificate where it is hardest: exponentials so far below a loose reference that they
are flushed to zero, and scores so close that no block is certain."""
import numpy as np
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_indices

pytestmark = pytest.mark.gpu


def _both(p):
    """The choice with the single-precision stages and with double precision everywhere."""
    import torch
    from paper_2512_13368_b200 import binding
    got = []
    for exact in (0, 1):
        binding.blossom_debug_switch(binding.SWITCH_EXACT_SELECT, exact)
        try:
            p.idx.fill_(-7)
            p.select()
            torch.cuda.synchronize()
            got.append(p.idx.cpu().numpy().copy())
        finally:
            binding.blossom_debug_switch(binding.SWITCH_EXACT_SELECT, -1)
    return got


@pytest.mark.parametrize("per_query", [0, 1])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_a_score_whose_exponential_is_flushed(dtype, per_query):
    """Two heads share a selection.  In the first the reference (69, from one long mean) lies so far above the
    logits that block 2's e^-18.4 is flushed; in the second nothing is, and there block 3 leads by less than the
    first head's loss.  Exactly, block 2 has 5.5e-9 and block 3 has 0.6e-9."""
    from paper_2512_13368_b200 import runner
    w = workloads.make("flushed", dtype, 1, 2, 80, 32, 16, 4, 16, seed=1, kv_heads=1)
    w.per_query = per_query
    w.q[:], w.k[:] = 0.0, 0.0
    w.q[0, 0, :, 1], w.q[0, 1, :, 2] = 1.0, 0.32421875
    w.k[0, 0, 16:32, 0] = 69.0
    w.k[0, 0, 32:48, 1], w.k[0, 0, 32:48, 2] = -18.375, -66.0
    w.k[0, 0, 48:64, 1], w.k[0, 0, 48:64, 2] = -22.0, -64.0
    p = runner.DeviceProblem(w, sm_scale=1.0)
    rows = slice(64, 80) if per_query else slice(4, 5)
    for got in _both(p):
        assert (got[0, 0, rows] == [0, 1, 2, 4]).all(), got[0, 0, rows]
    check_indices(w, got, sm_scale=1.0)


@pytest.mark.parametrize("length", [8.0, 20.0, 40.0, 60.0, 80.0, 120.0])
@pytest.mark.parametrize("H,Hkv,dtype,per_query", [(4, 2, "bf16", 0), (4, 2, "bf16", 1), (2, 2, "fp32", 0), (4, 1, "fp32", 1)])
def test_references_far_above_the_logits(length, H, Hkv, dtype, per_query):
    """Every norm bound is `length` (natural units) above logits that spread over twenty."""
    from paper_2512_13368_b200 import runner
    w = workloads.make("far", dtype, 2, H, 420, 32, 16, 5, 16, seed=int(length), lengths=(200, 420),
                       kv_heads=Hkv if Hkv != H else 0)
    w.per_query = per_query
    w.q[..., :2] = 0.0
    w.q /= np.linalg.norm(w.q, axis=-1, keepdims=True)
    w.k[:] = 0.0
    rng = np.random.default_rng(7)
    for b in range(27):     # a mean of its own per block
        m = rng.standard_normal((2, Hkv, 1, 32)).astype(np.float32) * 5.0
        m[..., 0] = length
        w.k[:, :, 16 * b:16 * (b + 1)] = m
    w.q, w.k = workloads.quantize(w.q, dtype), workloads.quantize(w.k, dtype)
    a, b = _both(runner.DeviceProblem(w, sm_scale=1.0))
    assert np.array_equal(a, b)
    check_indices(w, a, sm_scale=1.0)


@pytest.mark.parametrize("B,H,Hkv,L,D,block,dtype,opts", [
    (2, 2, 2, 640, 32, 16, "bf16", {}),         # decided inside the scoring kernel
    (2, 4, 2, 500, 32, 32, "bf16", {}),
    (2, 2, 2, 700, 32, 64, "fp32", {"causal": 0}),
    (2, 2, 2, 520, 32, 32, "bf16", {"cmp": (64, 32)}),
    (2, 2, 2, 1024, 64, 32, "bf16", {}),        # decided from the list
])
def test_scores_that_no_bound_separates(B, H, Hkv, L, D, block, dtype, opts):
    """Queries of 1e-5: every probability is 1 / n to six digits, so every block goes to double precision."""
    from paper_2512_13368_b200 import runner
    w = workloads.make("close", dtype, B, H, L, D, block, 4, 16, seed=L, lengths=(L // 2, L),
                       kv_heads=Hkv if Hkv != H else 0)
    w.causal = opts.get("causal", 1)
    w.cmp_block, w.cmp_stride = opts.get("cmp", (0, 0))
    w.q = workloads.quantize(w.q * np.float32(1e-5), dtype)
    a, b = _both(runner.DeviceProblem(w))
    assert np.array_equal(a, b)


@pytest.mark.parametrize("H,Hkv,L,block,dtype", [(2, 1, 8 * 1024, 8, "bf16"), (5, 1, 16 * 655, 16, "bf16"),
                                                 (5, 1, 16 * 670, 16, "bf16"), (1, 1, 16 * 1024, 16, "fp32")])
def test_per_position_selection_of_very_many_blocks(H, Hkv, L, block, dtype):
    """Around the number of blocks from which a warp keeps one head's logits at a time, and the largest number."""
    import torch
    from paper_2512_13368_b200 import binding, runner
    w = workloads.make("many", dtype, 1, H, L, 32, block, 4, 16, seed=H, kv_heads=Hkv if Hkv != H else 0)
    w.per_query = 1
    p = runner.DeviceProblem(w, training=False)
    p.select()
    torch.cuda.synchronize()
    check_indices(w, p.idx.cpu().numpy())
    assert binding.blossom_device_status(p.workspace) == 0
