"""The native half of the autograd front end: calls without a gradient, partial gradients, repeated
backwards, and what it refuses."""
import pytest

from paper_2512_13368_b200 import build


def test_host_tensors_are_refused_with_the_reason():
    import torch
    build.build()
    from paper_2512_13368_b200.autograd import blossom_attention
    q = torch.zeros(1, 2, 32, 32)
    with pytest.raises(ValueError):
        blossom_attention(q, q, q, torch.zeros(2, 2), 16, 2, 8)
    with pytest.raises(TypeError):
        blossom_attention(q.double(), q.double(), q.double(), torch.zeros(2, 2), 16, 2, 8)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,L,lens", [("bf16", 33, None), ("bf16", 300, "int64"), ("fp32", 70, "int32")])
def test_calls_without_a_gradient_and_partial_gradients(dtype, L, lens):
    import torch
    from paper_2512_13368_b200.autograd import blossom_attention
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(L)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    q, k, v = (mk(3, 2, L, 32).to(dt).requires_grad_(True) for _ in range(3))
    gate, dout = mk(2, 2).requires_grad_(True), mk(3, 2, L, 32).to(dt)
    n = None if lens is None else torch.tensor([L, 1, L // 2], dtype=getattr(torch, lens), device="cuda")
    call = lambda *a: blossom_attention(*a, 16, 3, 9, seq_lens=n, return_indices=True)  # noqa: E731
    out, idx = call(q, k, v, gate)
    assert out.requires_grad and not idx.requires_grad
    full = torch.autograd.grad(out, (q, k, v, gate), dout, retain_graph=True)
    again = torch.autograd.grad(out, (q, k, v, gate), dout)
    assert all(torch.equal(a, b) for a, b in zip(full, again))
    with pytest.raises(RuntimeError):   # the graph has been released
        torch.autograd.grad(out, (q,), dout)
    with torch.no_grad():
        out2, idx2 = call(q, k, v, gate)
    assert not out2.requires_grad and torch.equal(idx, idx2)   # (other kernels may serve it: not the same bits)
    assert torch.allclose(out.float(), out2.float(), rtol=1e-2, atol=1e-2 if dtype == "bf16" else 1e-5)
    d = [t.detach() for t in (q, k, v, gate)]
    for i in range(4):                  # only one input wants a gradient
        a = list(d)
        a[i] = d[i].clone().requires_grad_(True)
        o, _ = call(*a)
        (gi,) = torch.autograd.grad(o, (a[i],), dout)
        assert torch.equal(o, out) and torch.equal(gi, full[i])
    half = d[3].to(torch.bfloat16).requires_grad_(True)   # a gate stored in another type gets its gradient in it
    (gh,) = torch.autograd.grad(call(d[0], d[1], d[2], half)[0], (half,), dout)
    assert gh.dtype == torch.bfloat16
    with pytest.raises(ValueError):
        blossom_attention(d[0], d[1], d[2], mk(3, 2), 16, 3, 9)
    with pytest.raises(RuntimeError):   # BlossomError: the library does not take top_k = 0
        blossom_attention(*d, 16, 0, 9)


@pytest.mark.gpu
def test_transforms_without_a_rule_are_refused():
    """Batched tensors (vmap) and those of functional gradients have no memory that the library could read."""
    import torch
    from paper_2512_13368_b200.autograd import blossom_attention
    g = torch.Generator(device="cuda").manual_seed(1)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    q, k, v, gate = mk(2, 2, 70, 32), mk(2, 2, 70, 32), mk(2, 2, 70, 32), mk(2, 2)
    n = torch.tensor([70, 9], dtype=torch.int32, device="cuda")
    call = lambda a, b, c, d, e: blossom_attention(a, b, c, d, 16, 3, 9, seq_lens=e)  # noqa: E731
    args = [q, k, v, gate, n]
    for i, x in enumerate(args):
        f = lambda t: call(*args[:i], t, *args[i + 1:])  # noqa: E731,B023
        with pytest.raises(RuntimeError):
            torch.func.vmap(f)(torch.stack([x, x]))
        if i < 4:
            with pytest.raises(RuntimeError):
                torch.func.grad(lambda t: f(t).sum())(x)  # noqa: B023
    assert call(*args).shape == q.shape     # (and the interpreter is in order)


@pytest.mark.gpu
@pytest.mark.parametrize("train", [False, True])
def test_forward_mode_is_refused(train):
    """There is no forward-mode rule: a tangent is an error, never dropped."""
    import torch
    import torch.autograd.forward_ad as fwd
    from paper_2512_13368_b200.autograd import blossom_attention
    g = torch.Generator(device="cuda").manual_seed(1)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda").requires_grad_(train)  # noqa: E731
    args = [mk(2, 2, 70, 32), mk(2, 2, 70, 32), mk(2, 2, 70, 32), mk(2, 2)]
    with fwd.dual_level():
        for i in range(4):
            a = list(args)
            a[i] = fwd.make_dual(a[i], torch.ones_like(a[i]))
            with pytest.raises(NotImplementedError):
                blossom_attention(*a, 16, 3, 9)
    assert blossom_attention(*args, 16, 3, 9).shape == args[0].shape


@pytest.mark.gpu
@pytest.mark.parametrize("L,D,rope", [(70, 32, 0.0), (600, 64, 100.0)])
def test_everything_the_backward_needs_goes_through_the_saved_tensor_hooks(L, D, rope):
    """Offloaded to the host and brought back, or thrown away and computed again: the same gradients, and
    nothing of the call's size stays on the GPU between the passes."""
    import torch
    from torch.utils.checkpoint import checkpoint
    from paper_2512_13368_b200.autograd import blossom_attention
    g = torch.Generator(device="cuda").manual_seed(L)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    args = [mk(8, 2, L, D).bfloat16().requires_grad_(True) for _ in range(3)] + [mk(2, 2).requires_grad_(True)]
    dout = mk(8, 2, L, D).bfloat16()
    f = lambda *a: blossom_attention(*a, 32, 3, 40, rope_theta=rope)  # noqa: E731
    want = torch.autograd.grad(f(*args), args, dout)
    torch.cuda.synchronize()
    tensor = dout.nbytes

    def kept(make):
        before = torch.cuda.memory_allocated()
        out = make()
        return out, torch.cuda.memory_allocated() - before

    plain, size = kept(lambda: f(*args))
    assert size > 3 * tensor                # the output, both branches' rows, the workspace
    del plain
    with torch.autograd.graph.save_on_cpu():
        out, size = kept(lambda: f(*args))
    assert size < 2 * tensor                # the output alone
    for a, b in zip(want, torch.autograd.grad(out, args, dout, retain_graph=True)):
        assert torch.equal(a, b)
    for a, b in zip(want, torch.autograd.grad(out, args, dout)):
        assert torch.equal(a, b)
    del out
    out, size = kept(lambda: checkpoint(f, *args, use_reentrant=False))
    assert size < 2 * tensor
    for a, b in zip(want, torch.autograd.grad(out, args, dout)):
        assert torch.equal(a, b)
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t, lambda t: t[:1] if t.dtype == torch.uint8 else t):
        out = f(*args)
    with pytest.raises(RuntimeError):
        torch.autograd.grad(out, args, dout)


def test_layout_rules():
    import torch
    build.build()
    from paper_2512_13368_b200 import binding
    binding.load()
    from paper_2512_13368_b200 import _front
    x = torch.zeros(2, 3, 8, 32)
    for t, dense in ((x, True), (x.transpose(1, 2), True), (x.permute(3, 2, 0, 1), True), (x[:, :1], False),
                     (x[:1], True), (x[:, :, ::2], False), (x[:1].expand(2, 3, 8, 32), False), (x[:0], False),
                     (x[:, :, :1], False), (torch.zeros(5), True), (torch.zeros(5).expand(4, 5), False)):
        assert _front.dense(t) == dense, (t.shape, t.stride())
        if t.numel() and 0 not in t.stride():
            assert _front.like(t).stride() == t.stride() and _front.like(t).shape == t.shape
    for f in (_front.dense, _front.like):
        with pytest.raises(TypeError):
            f(3)


@pytest.mark.gpu
def test_every_layout_gives_what_the_dense_tensors_give():
    """Transposed, packed, strided and broadcast inputs, k and v in layouts of their own, transposed and
    broadcast upstream gradients; outputs and gradients keep the strides of a dense input."""
    import torch
    from paper_2512_13368_b200.autograd import blossom_attention
    B, H, L, D = 2, 3, 70, 32
    g = torch.Generator(device="cuda").manual_seed(5)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda").bfloat16()  # noqa: E731
    gate = torch.randn((H, 2), generator=g, device="cuda")

    def views(x):       # the same numbers [B, H, L, D] in other layouts
        yield x.transpose(1, 2).contiguous().transpose(1, 2)
        p = torch.zeros(B, L, 3, H, D, dtype=x.dtype, device="cuda")
        p[:, :, 1] = x.transpose(1, 2)
        yield p[:, :, 1].transpose(1, 2)
        w = torch.zeros(B, H, 2 * L, D, dtype=x.dtype, device="cuda")
        w[:, :, ::2] = x
        yield w[:, :, ::2]
        yield x.permute(3, 2, 1, 0).contiguous().permute(3, 2, 1, 0)    # the last dimension is not contiguous

    def step(q, k, v, dout):
        leaves = [t.detach().requires_grad_(True) for t in (q, k, v)]
        out = blossom_attention(*leaves, gate, 16, 3, 9)
        return [out.detach()] + list(torch.autograd.grad(out, leaves, dout))

    q, k, v, dout = mk(B, H, L, D), mk(B, H, L, D), mk(B, H, L, D), mk(B, H, L, D)
    want = step(q, k, v, dout)
    for i, x in enumerate((q, k, v, dout)):
        for t in views(x):
            a = [q, k, v, dout]
            a[i] = t
            assert torch.equal(t, x)
            got = step(*a)
            for y, z in zip(want, got):
                assert torch.equal(y, z), (i, t.stride())
    qt = next(views(q))
    assert step(qt, next(views(k)), next(views(v)), dout)[0].stride() == qt.stride()
    k1, d1 = mk(1, 1, L, D).expand(B, H, L, D), mk(1, 1, 1, D).expand(B, H, L, D)   # (strides of zero)
    for y, z in zip(step(q, k1.contiguous(), v, d1.contiguous()), step(q, k1, v, d1)):
        assert torch.equal(y, z)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,L,D", [("bf16", 70, 32), ("bf16", 450, 64), ("fp32", 70, 64)])
def test_negated_views_and_zero_tensors_in_a_layout_that_needs_no_copy(dtype, L, D):
    """Inputs and gradients that are dense, in q's own layout, but not plain memory: what plain copies give."""
    import torch
    from paper_2512_13368_b200.autograd import blossom_attention
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(L)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    B, H = 2, 3
    layouts = (lambda x: x, lambda x: x.transpose(1, 2).contiguous().transpose(1, 2))
    for layout in layouts:
        t = {n: layout(mk(B, H, L, D).to(dt)) for n in ("q", "k", "v", "dout")}
        t["gate"], t["phi"] = mk(H, 2), mk(16)
        t["lens"] = torch.tensor([L, L // 3], dtype=torch.int32, device="cuda")

        def step(a):
            leaves = [a[n].detach().requires_grad_(True) for n in ("q", "k", "v", "gate")]
            out, idx = blossom_attention(*leaves, 16, 3, 9, seq_lens=a["lens"], phi_logits=a["phi"], return_indices=True)
            with torch.no_grad():
                alone = blossom_attention(*(a[n] for n in ("q", "k", "v", "gate")), 16, 3, 9, seq_lens=a["lens"],
                                          phi_logits=a["phi"])
            return [out.detach(), idx, alone] + list(torch.autograd.grad(out, leaves, a["dout"]))

        want = step(t)
        for n, x in t.items():
            neg = torch._neg_view(-x)
            assert neg.is_neg() and torch.equal(neg, x) and neg.stride() == x.stride()
            for a, b in zip(want, step(dict(t, **{n: neg}))):
                assert torch.equal(a, b), n
            if n in ("lens", "phi"):
                continue
            zero = torch._efficientzerotensor(x.shape, dtype=x.dtype, device="cuda")
            if n != "gate" and layout is not layouts[0]:
                zero = torch._efficientzerotensor((B, L, H, D), dtype=dt, device="cuda").transpose(1, 2)
            assert zero._is_zerotensor()
            for a, b in zip(step(dict(t, **{n: torch.zeros_like(x)})), step(dict(t, **{n: zero}))):
                assert torch.equal(a, b), n
