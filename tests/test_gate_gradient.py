"""The gate gradient where both branches see the same keys (a window over the whole history and every
block selected): d alpha = sum (P_lt - P_st) dP is a sum of exact zeros, pair by pair, whatever the kernel,
tile order or reduction; formed as a sum per branch it would be the rounding that is left of two large
numbers."""
import numpy as np
import pytest

from paper_2512_13368_b200 import workloads

pytestmark = pytest.mark.gpu

SAME = [  # B, H, Hkv, L, D, block, lengths, options: the short kernels, then the tensor-core ones
    (4, 1, 1, 40, 64, 16, None, {}),
    (64, 2, 2, 50, 32, 16, (5, 50), {}),
    (3, 4, 2, 129, 64, 32, (7, 129), {}),
    (2, 2, 2, 80, 32, 16, None, {"causal": 0}),
    (300, 2, 2, 140, 64, 32, (1, 140), {}),   # short forward, tensor-core backward
    (3, 1, 1, 600, 64, 64, None, {}),
    (2, 3, 3, 777, 32, 32, (100, 777), {}),
    (2, 4, 2, 640, 64, 64, (65, 640), {}),    # a CTA's rows are two heads' positions
    (2, 2, 2, 520, 64, 16, (9, 520), {"causal": 0}),
    (2, 2, 1, 530, 32, 32, None, {"per_query": 1}),
    (2, 2, 2, 70, 32, 16, (3, 70), {"dtype": "fp32"}),
]


def _problem(B, H, Hkv, L, D, block, lens, opts, window):
    from paper_2512_13368_b200 import runner
    w = workloads.make("same-keys", opts.get("dtype", "bf16"), B, H, L, D, block, -(-L // block), window, seed=L + D,
                       lengths=lens, kv_heads=Hkv if Hkv != H else 0)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    p = runner.DeviceProblem(w)
    p.step()
    return w, p.results()


@pytest.mark.parametrize("B,H,Hkv,L,D,block,lens,opts", SAME)
def test_branches_that_see_the_same_keys_leave_exactly_no_gate_gradient(B, H, Hkv, L, D, block, lens, opts):
    w, res = _problem(B, H, Hkv, L, D, block, lens, opts, L)
    assert np.array_equal(res["lse"][0], res["lse"][1])
    assert not res["dgate"].any(), res["dgate"]


@pytest.mark.parametrize("L,D,block", [(48, 64, 16), (200, 32, 16), (600, 64, 64)])
def test_a_window_one_key_short_of_the_history(L, D, block):
    """Only the last row's branches differ, by its first key.  Its probabilities carry the rounding of an
    exponent of at most 2^5 in log2 units (2^-19, and as much for the log-sum-exp and the exponential); the
    other rows add nothing, so the bar does not grow with their number."""
    import oracle
    w, res = _problem(3, 1, 1, L, D, block, None, {}, L - 1)
    ref = oracle.forward_backward(w.q, w.k, w.v, w.gate, w.dout, block, -(-L // block), L - 1, idx=res["idx"])
    a = 1.0 / (1.0 + np.exp(-(float(w.gate[0, 0]) - float(w.gate[0, 1]))))
    q, k, v, g = (x.astype(np.float64)[:, 0] for x in (w.q, w.k, w.v, w.dout))
    z = np.einsum("nd,npd->np", q[:, -1], k) / np.sqrt(D)
    assert np.abs(z).max() * np.log2(np.e) < 32
    pl = np.exp(z - z.max(1, keepdims=True))
    ps = pl.copy()
    ps[:, 0] = 0.0
    dp = np.abs(np.einsum("nd,npd->np", g[:, -1], v))
    size = a * (1 - a) * ((pl / pl.sum(1, keepdims=True) + ps / ps.sum(1, keepdims=True)) * dp).sum()
    err = np.abs(res["dgate"].astype(np.float64) - ref["dgate"]).max()
    print(err / size)
    assert err <= 3 * 2.0 ** -19 * size
