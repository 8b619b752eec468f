"""Rows copied between layouts: the front end's way from a view to the layout that the kernels want."""
import ctypes

import pytest

from paper_2512_13368_b200 import binding, build


def copy_rows(src, dst, stream=None):
    """`src` into `dst` ([B, H, L, D] CUDA tensors); the status."""
    e = src.element_size()
    strides = lambda t: (ctypes.c_int64 * 3)(*(t.stride(i) * e for i in range(3)))  # noqa: E731
    return binding.load().blossom_copy_rows(*src.shape[:3], src.shape[3] * e, ctypes.c_void_p(src.data_ptr()), strides(src),
                                            ctypes.c_void_p(dst.data_ptr()), strides(dst), ctypes.c_void_p(stream))


def test_what_is_not_in_whole_pieces_is_refused():
    build.build()
    lib = binding.load()
    s = (ctypes.c_int64 * 3)(1024, 512, 64)
    call = lambda B=1, H=2, L=8, n=64, src=4096, a=s, dst=8192, b=s: lib.blossom_copy_rows(  # noqa: E731
        B, H, L, n, ctypes.c_void_p(src), a, ctypes.c_void_p(dst), b, None)
    bad = lambda *x: (ctypes.c_int64 * 3)(*x)  # noqa: E731
    for kw in (dict(B=0), dict(H=-1), dict(L=0), dict(src=None), dict(dst=None), dict(a=None), dict(b=None)):
        assert call(**kw) == 1, kw
    for kw in (dict(n=0), dict(n=8), dict(n=48), dict(n=72), dict(n=8192), dict(src=4104), dict(dst=8196),
               dict(a=bad(1024, 512, 72)), dict(b=bad(1024, 520, 64)), dict(a=bad(-1024, 512, 64)), dict(B=1 << 20, L=1 << 20)):
        assert call(**kw) == 2, kw


@pytest.mark.parametrize("B,H,L", [(1 << 22, 1 << 22, 1 << 20),             # 2^64 rows: 0 in 64 bits
                                   (1 << 22, 1 << 21, (1 << 21) + 1),       # 2^64 + 2^43
                                   ((1 << 31) - 1, (1 << 31) - 1, (1 << 31) - 1),
                                   (1 << 15, 1 << 15, 2)])                  # 2^31
def test_more_rows_than_64_bits_count_are_refused(B, H, L):
    build.build()
    s = (ctypes.c_int64 * 3)(1024, 512, 64)
    assert binding.load().blossom_copy_rows(B, H, L, 64, ctypes.c_void_p(4096), s, ctypes.c_void_p(8192), s, None) == 2


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,L,D", [(1, 1, 1, 8), (2, 3, 5, 32), (1, 1, 255, 32), (1, 2, 129, 64), (3, 300, 1, 32),
                                     (70, 7, 3, 64), (2, 2, 33, 2048), (5, 2, 1024, 32)])
def test_every_order_of_the_dimensions(B, H, L, D):
    import torch
    x = torch.randn(B, H, L, D, device="cuda").bfloat16()
    orders = [(0, 1, 2), (0, 2, 1), (2, 1, 0), (1, 0, 2)]

    def laid_out(order, fill):
        gap = torch.full([x.shape[i] for i in order] + [D + 8], fill, dtype=x.dtype, device="cuda")
        back = [order.index(i) for i in range(3)] + [3]
        return gap, gap[..., :D].permute(back)
    for a in orders:
        _, src = laid_out(a, 0.0)
        src.copy_(x)
        for b in orders:
            gap, dst = laid_out(b, 7.0)
            assert copy_rows(src, dst) == 0
            assert torch.equal(dst, x) and (gap[..., D:] == 7).all()    # nothing beside the rows
    dst = torch.empty_like(x)
    assert copy_rows(x[:1, :, :1].expand(B, H, L, D), dst) == 0         # strides of zero repeat
    assert torch.equal(dst, x[:1, :, :1].expand(B, H, L, D))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,D", [("bf16", 32), ("fp32", 64)])
def test_gradients_that_are_not_plain_memory(dtype, D):
    """Transposed negated views and zero tensors (those in the output's own layout are in test_front_native.py), misaligned
    and repeated rows: what their plain copies give."""
    import torch
    from paper_2512_13368_b200.autograd import blossom_attention
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(D)
    mk = lambda *s: torch.randn(s, generator=g, device="cuda").to(dt)  # noqa: E731
    B, H, L = 2, 2, 40
    q, k, v = (mk(B, H, L, D).requires_grad_(True) for _ in range(3))
    gate = torch.randn((H, 2), generator=g, device="cuda").requires_grad_(True)
    out = blossom_attention(q, k, v, gate, 16, 2, 9)
    grads = lambda d: torch.autograd.grad(out, (q, k, v, gate), d, retain_graph=True)  # noqa: E731
    x = mk(B, L, H, D).transpose(1, 2)
    flat = torch.zeros(B * L * H * D + 1, dtype=dt, device="cuda")
    odd = flat[1:].view(B, L, H, D).transpose(1, 2)      # rows that start off a 16-byte boundary
    odd.copy_(x)
    for d in (torch._neg_view(x), torch._efficientzerotensor((B, L, H, D), dtype=dt, device="cuda").transpose(1, 2),
              odd, x[:, :, :1].expand(B, H, L, D)):
        plain = torch.empty(B, H, L, D, dtype=dt, device="cuda").copy_(d)
        for a, b in zip(grads(plain), grads(d)):
            assert torch.equal(a, b)
