"""Bytes of the tile lists: a kernel holds those that it reads in shared memory, beside what decides how many of its CTAs share an
SM, so an image has no parts that nobody reads.  Two images (query-major, key-major) per 128 rows are all of the
workspace that grows with the square of the length."""
import pytest

from paper_2512_13368_b200 import binding, build


@pytest.mark.parametrize("heads,kv_heads", [(1, 1), (4, 4), (4, 1)])
def test_bytes_per_tile(heads, kv_heads):
    build.build()
    step = 16384  # a multiple of everything that a part is rounded to

    def size(x):
        return binding.blossom_workspace_bytes(binding.make_params(1, heads, x * step, 64, 64, 16, 256, "bf16", kv_heads=kv_heads))

    quadratic = (size(3) - 2 * size(2) + size(1)) / 2
    tiles, images = step // 64, step // 128
    # query-major: lists 6 and classes 16 for dQ, selections 8, items 8 and classes 8 for the forward; key-major: 6 + 16 + 8
    # (there is room for a key-major image per query head, however many key/value heads there are)
    assert quadratic <= images * tiles * heads * (46 + 30) * 1.001
