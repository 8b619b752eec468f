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
