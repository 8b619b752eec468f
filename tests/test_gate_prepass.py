"""The input-dependent gate's pre-pass with several rows a thread: one, two and four passes, a last part
that is ragged or only the padding of L to 64, query blocks larger than a pass, and lengths that leave
whole parts without a row.  Against the oracle; repeated calls give the same bits."""
import numpy as np
import pytest

from paper_2512_13368_b200 import workloads
from parity_util import check_forward_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,L,D,block,lens,rows", [
    (2, 2, 65, 64, 64, (0, 65), 64),        # one pass of 32 rows, but blocks of 64
    (37, 2, 257, 64, 32, (1, 257), 64),     # 666 passes: two a CTA, the last part one row and its padding
    (75, 2, 250, 64, 16, (20, 250), 128),    # 1200: four a CTA, the second part ragged
    (100, 4, 129, 32, 16, (3, 129), 256),    # 1200 passes of 64 rows
    (148, 2, 33, 64, 32, None, 64),         # 592: two a CTA
])
def test_several_rows_a_thread(B, H, L, D, block, lens, rows):
    import torch
    from paper_2512_13368_b200 import binding, runner
    w = workloads.make("gate-prep", "bf16", B, H, L, D, block, 2, 20, seed=L, lengths=lens)
    w.gate_mode = 1
    w.gate = (0.3 * np.random.default_rng(L).standard_normal((H, 2 * D + 1))).astype(np.float32)
    p = runner.DeviceProblem(w)
    assert binding.blossom_launch_plan(p.params, binding.PLAN_GATE_ROWS, lens is not None) == rows   # of a CTA
    p.step()
    print(check_forward_backward(w, p.results()))
    first = {k: getattr(p, k).clone() for k in ("dq", "dk", "dv", "dgate")}
    p.backward()
    for k, t in first.items():
        assert torch.equal(t, getattr(p, k)), k
