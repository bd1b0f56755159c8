"""A workspace that is large enough for a call is large enough for every smaller one:
callers size it once for their largest (CPU only)."""
import itertools

import pytest

from paper_2506_05558_gb300 import gs


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


EDGES = [0, 1, 2047, 2048, 2049, 4095, 4096, 4097, 200_000, 622_592, 622_593, 1_000_000, (1 << 20) - 1, 1 << 20,
         (1 << 20) + 1, (1 << 20) + 4096, 1_090_000, 1 << 21, (1 << 21) + 1, 4 << 20, (4 << 20) + 1, 5 << 20]


@pytest.mark.parametrize("frame", [[(64, 64)], [(1920, 1080)], [(640, 480)] * 4])
def test_sort_workspace_grows_with_items_and_capacity(frame):
    f = gs.frame(frame)
    size = {(n, c): gs.gs_sort_workspace_size(n, f, c) for n in EDGES for c in EDGES}
    for (a, b), k in itertools.product(zip(EDGES, EDGES[1:]), EDGES):
        assert size[a, k] <= size[b, k], (a, b, k)
        assert size[k, a] <= size[k, b], (k, a, b)


def test_sort_workspace_grows_with_tiles():
    # around 2^20 tiles of 8 pixels
    for n, c in ((0, 0), (1000, 5000), (1 << 20, 1 << 20)):
        sizes = [gs.gs_sort_workspace_size(n, gs.frame([(8 * w, 8 * 1024)], 8), c) for w in (1, 500, 1023, 1024, 1025, 1100, 2049)]
        assert sizes == sorted(sizes)


def test_spawn_workspace_depends_on_the_pixels_alone():
    sizes = [gs.gs_spawn_workspace_size(w, h) for w, h in ((1920, 1080), (1080, 1920), (2073600, 1), (1, 2073600), (33, 62836))]
    assert all(s <= sizes[0] for s in sizes), sizes
    grow = [gs.gs_spawn_workspace_size(w, h) for w, h in ((1, 1), (31, 1), (1, 32), (64, 64), (65, 64), (31, 4000), (4000, 32))]
    assert grow == sorted(grow), grow
