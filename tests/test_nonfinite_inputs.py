"""Queries and keys that are not finite (a diverged model): the index rows stay rows - the own block once,
ascending, in range, as many as fit - nothing outside the index array is written, and sequences that hold
finite numbers get what they get without their neighbours."""
import numpy as np
import pytest

from paper_2512_13368_b200 import workloads

pytestmark = pytest.mark.gpu

CASES = [  # dtype, H, Hkv, L, D, block, topk, options: each names a stage that decides in double precision
    ("bf16", 2, 2, 1024, 64, 32, 4, {}),                    # a list of blocks
    ("fp32", 2, 2, 500, 64, 16, 4, {}),
    ("bf16", 2, 2, 600, 32, 16, 3, {}),                     # inside the scoring kernel
    ("bf16", 2, 2, 600, 32, 32, 3, {"causal": 0}),
    ("bf16", 1, 1, 2400, 64, 16, 5, {}),                    # more than 128 blocks
    ("fp32", 1, 1, 2400, 32, 16, 5, {"causal": 0}),
    ("bf16", 4, 2, 300, 32, 8, 4, {}),                      # blocks of 8
    ("bf16", 4, 2, 640, 64, 32, 4, {"cmp": (64, 16)}),
    ("bf16", 4, 2, 400, 64, 16, 4, {"per_query": 1}),       # a position at a time
    ("fp32", 2, 2, 300, 32, 16, 4, {"per_query": 1}),
    ("bf16", 1, 1, 2200, 32, 16, 4, {"per_query": 1}),
    ("bf16", 2, 2, 200, 32, 16, 4, {}),                     # the short-history kernel
    ("bf16", 8, 2, 200, 64, 16, 4, {"cmp": (32, 16)}),
    ("bf16", 2, 2, 143, 64, 32, 2, {"causal": 0}),
]


@pytest.mark.parametrize("where", ["query", "key", "both"])
@pytest.mark.parametrize("dtype,H,Hkv,L,D,block,topk,opts", CASES)
def test_index_rows_of_non_finite_inputs(dtype, H, Hkv, L, D, block, topk, opts, where):
    import torch
    from paper_2512_13368_b200 import runner
    w = workloads.make("non-finite", dtype, 6, H, L, D, block, topk, 20, seed=L, lengths=(L // 2, L),
                       kv_heads=Hkv if Hkv != H else 0)
    w.causal, w.per_query = opts.get("causal", 1), opts.get("per_query", 0)
    w.cmp_block, w.cmp_stride = opts.get("cmp", (0, 0))
    p = runner.DeviceProblem(w, training=False)
    p.forward()
    want, out = p.idx.clone(), p.out.clone()
    n = p.idx.numel()
    guarded = torch.full((n + 4096,), -7, dtype=torch.int32, device=p.idx.device)
    p.idx = guarded[:n].view(p.idx.shape)
    nan, inf = float("nan"), float("inf")
    t = L - L // 3
    if where != "key":
        p.q[1] = nan
        p.q[2, :, t] = nan
        p.q[3, :, t, 1] = inf
        p.q[5, :, -1, 0] = -inf
    if where != "query":
        p.k[1] = nan
        p.k[2, :, t, 3] = nan
        p.k[3, :, t, 3] = inf
        p.k[5, :, -block - 1] = -inf
    rows = w.L if w.per_query else w.n_blocks
    for call in (p.forward, p.select):      # (the attention's own entry and the selection's)
        guarded.fill_(-7)
        call()
        torch.cuda.synchronize()
        assert bool((guarded[n:] == -7).all())
        idx = p.idx.cpu().numpy()
        for seq in range(w.B):
            first = (w.L - int(w.seq_lens[seq])) // block
            for h in range(Hkv):
                for r in range(rows):
                    own = r // block if w.per_query else r
                    got = idx[seq, h, r]
                    kept = got[got >= 0]
                    padded = r < w.L - w.seq_lens[seq] if w.per_query else (r + 1) * block <= w.L - w.seq_lens[seq]
                    if padded:
                        assert (got == -1).all()
                        continue
                    last = own if w.causal else w.n_blocks - 1
                    assert (got[len(kept):] == -1).all() and (np.diff(kept) > 0).all() and own in kept, (seq, h, r, got)
                    assert kept[0] >= first and kept[-1] <= last, (seq, h, r, got)
                    assert len(kept) == min(topk, last - first + 1), (seq, h, r, got)
        for seq in (0, 4):
            assert torch.equal(p.idx[seq], want[seq]) and torch.equal(p.out[seq], out[seq])
