"""gs_sort in one CTA: inputs at both sides of its rule (4096 items, 256 tiles, 24576 possible
pairs or as many by the capacity) against stable sorts in PyTorch, bit for bit."""
import pytest
import torch

from paper_2506_05558_gb300 import gs
from test_gpu_sort_edges import built, check, projected  # noqa: F401  (built: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sizes,tile,rect_max,visible,levels,huge,caps", [
    (2048, [(48, 64)], 16, 3, 1.0, 1 << 20, 300, (1 << 20, 5000, 1)),   # 24576 possible pairs
    (2049, [(48, 64)], 16, 3, 1.0, 1 << 20, 300, (1 << 20, 24576)),     # more: general, and by capacity
    (4096, [(64, 48)], 16, 4, 1.0, 7, 4096, (24576, 24577)),            # every rect its view, cut
    (4097, [(16, 16)], 16, 1, 1.0, 1 << 20, 0, (1 << 20,)),
    (4096, [(16, 16)], 16, 1, 1.0, 1, 0, (1 << 20, 4096, 4095)),        # one tile, one depth
    (96, [(256, 256)], 16, 16, 0.9, 50, 20, (1 << 20, 3000)),           # 256 tiles
    (95, [(257, 256)], 16, 16, 0.9, 50, 20, (1 << 20,)),
    (512, [(64, 64), (33, 17), (16, 16), (8, 8)], 8, 4, 0.7, 1 << 20, 9, (20000, 700)),
    (1023, [(64, 64)], 16, 4, 0.0, 3, 0, (1 << 20,)),
    (1025, [(64, 64)], 16, 4, 0.5, 1 << 20, 0, (1 << 20,)),
])
def test_sort_small(n, sizes, tile, rect_max, visible, levels, huge, caps):
    f, p = projected(n, sizes, tile, rect_max, n + 1, visible, levels, huge)
    for cap in caps:
        check(n, f, p, cap)


def test_sort_small_wide_depths():
    """Depths over the whole range of positive floats: every digit of the keys in use."""
    n = 3000
    f, p = projected(n, [(40, 30)], 16, 2, 3, visible=1.0)
    bits = torch.randint(1, 0x7F800000, (n,), generator=torch.Generator().manual_seed(1), dtype=torch.int32)
    p.rgb_depth[:, 3] = bits.view(torch.float32).cuda()
    check(n, f, p, 1 << 16)


def test_sort_small_items_without_tiles():
    n = 1000
    f, p = projected(n, [(64, 64)], 16, 4, 5, visible=1.0)
    hollow = torch.rand(n, generator=torch.Generator().manual_seed(2)) < 0.3
    p.rect[hollow.cuda(), 2] = p.rect[hollow.cuda(), 0]
    check(n, f, p, 40000, emit=False)
