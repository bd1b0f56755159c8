"""gs_sort against stable sorts in PyTorch (whole numbers, bit for bit) at the edges of
its launches: radix tiles of 4096 keys and look-back groups of 16 of them, chunks of
2048 items, groups of 32 items, spans of 1024 pairs, rects of one tile and of the whole
view, equal depths, one and several digits of tile index, cut capacities."""
import numpy as np
import pytest
import torch

from paper_2506_05558_gb300 import gs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


def projected(n, sizes, tile, rect_max, seed, visible=0.7, levels=1 << 20, huge=0):
    """Random rects and depths for n items in each view; `huge` items cover their view."""
    rng = np.random.default_rng(seed)
    f = gs.frame(sizes, tile)
    nv = len(sizes)
    tx, ty = np.array(f.tiles_x[:nv]), np.array(f.tiles_y[:nv])
    v = np.repeat(np.arange(nv), n)
    x0 = (rng.random(nv * n) * tx[v]).astype(np.int64)
    y0 = (rng.random(nv * n) * ty[v]).astype(np.int64)
    x1 = np.minimum(x0 + rng.integers(1, rect_max + 1, nv * n), tx[v])
    y1 = np.minimum(y0 + rng.integers(1, rect_max + 1, nv * n), ty[v])
    big = rng.permutation(nv * n)[:huge]
    x0[big] = y0[big] = 0
    x1[big], y1[big] = tx[v[big]], ty[v[big]]
    see = rng.random(nv * n) < visible
    depth = (0.2 + rng.integers(0, levels, nv * n) * (50.0 / levels)).astype(np.float32)
    p = gs.Projected.alloc(nv * n)
    rgbd = np.zeros((nv * n, 4), np.float32)
    rgbd[:, 3] = depth
    p.rgb_depth.copy_(torch.from_numpy(rgbd))
    p.rect.copy_(torch.from_numpy(np.stack([x0, y0, x1, y1], 1).astype(np.uint16).view(np.int16)))
    p.n_tiles.copy_(torch.from_numpy(np.where(see, (x1 - x0) * (y1 - y0), 0).astype(np.int32)))
    return f, p


def reference(p, n, f, capacity):
    r = p.rect.cpu().numpy().view(np.uint16).astype(np.int64)
    nt = p.n_tiles.cpu().numpy().astype(np.int64)
    d = p.rgb_depth[:, 3].cpu().numpy().view(np.uint32)
    items = np.nonzero(nt > 0)[0]
    items = items[np.argsort(d[items], kind="stable")]
    w, h = r[items, 2] - r[items, 0], r[items, 3] - r[items, 1]
    cnt = w * h
    src = np.repeat(items, cnt)
    local = np.arange(cnt.sum()) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    ww = np.repeat(w, cnt)
    v = src // n
    tiles_x, base = np.array(f.tiles_x[:f.n_views]), np.array(f.tile_base[:f.n_views])
    t = base[v] + (r[src, 1] + local // np.maximum(ww, 1)) * tiles_x[v] + r[src, 0] + local % np.maximum(ww, 1)
    offset = np.cumsum(np.maximum(nt, 0)) - np.maximum(nt, 0)
    total = len(src)
    t, src, slot = t[:capacity], src[:capacity], (offset[src] + local)[:capacity]
    o = np.argsort(t, kind="stable")
    n_all = f.tile_base[f.n_views]
    lo, hi = np.searchsorted(t[o], np.arange(n_all), "left"), np.searchsorted(t[o], np.arange(n_all), "right")
    rng = np.where((hi > lo)[:, None], np.stack([lo, hi], 1), 0)
    order = np.argsort(-np.minimum(hi - lo, 0xFFFF), kind="stable")
    return total, src[o], slot[o], offset, rng, order


def check(n, f, p, capacity, emit=True):
    n_all = f.tile_base[f.n_views]
    out = gs.Pairs.alloc(n * f.n_views, n_all, capacity)
    for t in (out.src, out.emit, out.offset, out.range, out.order):
        t.fill_(-7)
    ws = gs.workspace(gs.gs_sort_workspace_size(n, f, out.capacity))
    ws.fill_(0x5A)  # nothing in it may have to start at zero
    gs.gs_sort(p, n, f, out, ws)
    torch.cuda.synchronize()
    total, src, slot, offset, rng, order = reference(p, n, f, out.capacity)
    k = min(total, out.capacity)
    assert int(out.count.item()) == total
    assert int(out.status.item()) == (gs.GS_ERR_CAPACITY if total > out.capacity else gs.GS_OK)
    i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a).astype(np.int32))
    assert torch.equal(out.offset.cpu()[:len(offset)], i32(offset))
    assert torch.equal(out.range.cpu().view(-1, 2), i32(rng))
    assert torch.equal(out.src.cpu()[:k], i32(src))
    if emit:
        assert torch.equal(out.emit.cpu()[:k], i32(slot))
    assert torch.equal(out.order.cpu(), i32(order))
    return total


@pytest.mark.parametrize("n,sizes,tile,rect_max,visible,levels,huge", [
    (1, [(16, 16)], 16, 1, 1.0, 1, 0),
    (31, [(64, 48)], 16, 4, 0.0, 9, 0),
    (33, [(64, 48)], 16, 4, 1.0, 1, 0),
    (256, [(1024, 16)], 16, 3, 1.0, 5, 1),
    (2048, [(256, 256), (17, 33)], 16, 2, 1.0, 1 << 20, 0),
    (2049, [(333, 257)], 8, 9, 0.7, 100, 3),
    (4096, [(640, 480)], 32, 1, 1.0, 1 << 20, 0),
    (4097, [(640, 480), (64, 64), (1, 1)], 16, 3, 1.0, 1 << 20, 0),
    (65536, [(1920, 1080)], 16, 1, 1.0, 1 << 20, 0),
    (65537, [(1920, 1080)], 16, 1, 1.0, 2, 40),
    (150001, [(1920, 1080), (720, 405)], 8, 2, 0.6, 1 << 20, 5),
    (1300000, [(1280, 720)], 16, 2, 0.9, 1 << 20, 0),
])
def test_sort_edges(n, sizes, tile, rect_max, visible, levels, huge):
    f, p = projected(n, sizes, tile, rect_max, n, visible, levels, huge)
    total = check(n, f, p, 1 << 16 if n < 4000 else 8 * n * len(sizes) + 400000)
    for cap in {max(total, 1), max(total - 1, 1), max(total // 2, 1), min(max(total, 1), 1024), 1}:
        if n < 200000 or cap == total // 2:
            check(n, f, p, cap)


def test_visible_items_without_tiles():
    """Items marked visible whose rect is empty (input not from gs_project) give no pairs."""
    n = 3000
    f, p = projected(n, [(500, 300)], 16, 4, 5, visible=1.0)
    hollow = torch.rand(n, generator=torch.Generator().manual_seed(2)) < 0.3
    p.rect[hollow.cuda(), 2] = p.rect[hollow.cuda(), 0]
    check(n, f, p, 40000, emit=False)
