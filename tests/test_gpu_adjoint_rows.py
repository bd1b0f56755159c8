"""The adjoint by rows of pixels (launches of 3,040 tiles and more) against the kernel of
small launches, which takes the tiles with long lists of such launches too: geometric
gradients bit for bit, colour and opacity sums up to the order of their additions, each
against the sum of its own terms' magnitudes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2506_05558_gb300 import gs, synth  # noqa: E402
from paper_2506_05558_gb300.raster import Rasterizer  # noqa: E402
from test_gpu_render_paths import run, scene  # noqa: E402

BG = (0.3, 0.1, 0.7)


def gradient(size):
    gen = torch.Generator(device="cuda").manual_seed(5)
    return torch.randn(3 * size[0] * size[1], generator=gen, device="cuda")


def compare(one, d_one, many, d_many, d_abs, tiles):
    """One view in a small launch against its copies in a large one."""
    for a, b in zip(one, many):
        for v in range(len(b)):
            assert torch.equal(a[0], b[v])
    # additions a colour term passes through: 8 in a row, 3 over rows and halves, 8 over blocks
    # and one per tile of its Gaussian; each rounds by 2^-24 of the partial sum
    steps = 19 + tiles
    for d in d_many:
        assert torch.equal(d_one[0, :, :5], d[:, :5])
        assert ((d_one[0, :, 6:] - d[:, 6:]).abs() <= 2 * steps * 2.0 ** -24 * d_abs[0, :, 6:]).all()


@pytest.mark.parametrize("kind,n,size,schedule", [
    ("plain", 6000, (403, 301), 0), ("plain", 6000, (404, 304), 1), ("opaque", 20000, (403, 301), 2),
    ("opaque", 3, (403, 301), 0), ("thin", 4000, (403, 301), 0), ("large", 3000, (404, 303), 0)])
def test_rows_match_small_launch(kind, n, size, schedule):
    sc, cam = scene(kind, n, size)
    dL = gradient(size)
    one, d_one = run(sc, cam, 1, schedule, dL, BG)
    many, d_many = run(sc, cam, 7, schedule, dL, BG)  # 3,458 tiles
    _, d_abs = run(sc, cam, 1, schedule, dL.abs(), BG)
    compare(one, d_one, many, d_many, d_abs, 494)


def clustered(n, in_cluster, logit, size):
    """n Gaussians all over the view and in_cluster more in 90 x 90 pixels of it."""
    w, h = size
    rng = np.random.default_rng(9)
    z = rng.uniform(3, 20, n + in_cluster)
    uv = np.concatenate([rng.uniform(-0.5, 0.5, (n, 2)) * [w, h], rng.uniform(-45, 45, (in_cluster, 2))])
    sc, cams, _ = synth.multiview_scene(seed=31, n=n + in_cluster, n_views=1, sizes=[size])
    f = 0.8 * w
    cam = synth.camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), f, w, h)
    sc.mean_opa[:, 0], sc.mean_opa[:, 1], sc.mean_opa[:, 2] = uv[:, 0] * z / f, uv[:, 1] * z / f, z
    sc.mean_opa[:, 3] = logit
    sc.scale[:, :3] = np.log(1.5 * z / f)[:, None]
    return sc, cam


# transparent: the long lists are composited to their ends; opaque: a few hundred entries of them;
# 33 views have 16,302 tiles, 34 more than the launches with long lists of their own
@pytest.mark.parametrize("logit,copies,schedule", [(-4.0, 7, 0), (1.0, 7, 0), (-4.0, 7, 1), (1.0, 13, 2), (-4.0, 33, 0), (-4.0, 34, 0)])
def test_long_lists_match_small_launch(logit, copies, schedule):
    size = (404, 301)
    sc, cam = clustered(6000, 20000, logit, size)
    dL = gradient(size)
    one, d_one = run(sc, cam, 1, schedule, dL, BG)
    many, d_many = run(sc, cam, copies, schedule, dL, BG)
    _, d_abs = run(sc, cam, 1, schedule, dL.abs(), BG)
    compare(one, d_one, many, d_many, d_abs, 494)


def test_long_lists_by_themselves():
    """What the rule counts as long is there, in graphs, on another stream and without a pair count
    (then no list is long) all the same gradients."""
    size, copies = (404, 301), 7
    sc, cam = clustered(6000, 20000, -4.0, size)
    g, cams = gs.Gaussians.from_scene(sc), gs.cameras_tensor([cam] * copies)
    r = Rasterizer(g.n, [size] * copies, 1 << 20)
    r.fit_capacity(g, cams)
    r.forward(g, cams)
    dL = gradient(size).repeat(copies)
    want = torch.zeros((copies, g.n, 9), device="cuda")
    r.backward(g, cams, dL, d_proj=want)
    torch.cuda.synchronize()
    lists = r.pairs.range.view(-1, 2)
    length = lists[:, 1] - lists[:, 0]
    long = length > max(1024, 8 * r.pair_count() / len(length))
    assert len(length) >= 3040 and 50 <= int(long.sum()) < len(length) // 2
    got = torch.zeros_like(want)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        r.backward(g, cams, dL, d_proj=got)
    torch.cuda.synchronize()
    assert torch.equal(want, got)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        r.backward(g, cams, dL, d_proj=got)
    for _ in range(5):
        got.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(want, got)
    count, r.pairs.count = r.pairs.count, None
    r.backward(g, cams, dL, d_proj=got)
    torch.cuda.synchronize()
    r.pairs.count = count
    assert torch.equal(want[..., :5], got[..., :5])


def opacity_magnitudes(r, v_size, dL, bg):
    """Per item the sum over pixels of |dL/dalpha| exp(-q/2) in 64 bits, from the projected rows."""
    w, h = v_size
    xy, co, rgbd = (t.double() for t in (r.proj.mean2d, r.proj.conic_opa, r.proj.rgb_depth))
    shown = r.proj.n_tiles[:r.n] > 0
    order = torch.nonzero(shown)[:, 0][torch.argsort(rgbd[:r.n][shown][:, 3])]
    y, x = torch.meshgrid(torch.arange(h, device="cuda") + 0.5, torch.arange(w, device="cuda") + 0.5, indexing="ij")
    dC = dL.double().view(3, h, w)
    T = torch.ones((h, w), device="cuda", dtype=torch.float64)
    live = torch.ones((h, w), device="cuda", dtype=torch.bool)
    steps = []
    for i in order.tolist():
        dx, dy = x - xy[i, 0], y - xy[i, 1]
        G = torch.exp(-0.5 * (co[i, 0] * dx * dx + 2 * co[i, 1] * dx * dy + co[i, 2] * dy * dy))
        a = torch.clamp(co[i, 3] * G, max=r.cfg.alpha_max)
        on = live & (a >= r.cfg.alpha_min)
        live &= ~(on & (T * (1 - a) < r.cfg.t_min))
        on &= live
        steps.append((i, G, torch.where(on, a, 0.0), T.clone()))
        T = torch.where(on, T * (1 - a), T)
    S = T * sum(dC[c] * bg[c] for c in range(3))
    out = torch.zeros((r.n,), device="cuda", dtype=torch.float64)
    for i, G, a, Tf in reversed(steps):
        gc = sum(dC[c] * rgbd[i, c] for c in range(3))
        dalpha = Tf * gc - S / (1 - a)
        out[i] = ((a > 0) * dalpha.abs() * G).sum()
        S = S + a * Tf * gc
    return out


def test_opacity_gradient_item_by_item():
    size, copies = (112, 112), 64  # 49 tiles a view, 3,136 in all
    sc, cam = scene("plain", 300, size)
    sc.scale[:, :3] += 1.0
    dL = gradient(size)
    cfg = gs.config(sh_degree=3, bg=BG)
    out = []
    for k in (1, copies):
        r = Rasterizer(sc.n, [size] * k, 1 << 16, cfg)
        g, cams = gs.Gaussians.from_scene(sc), gs.cameras_tensor([cam] * k)
        r.fit_capacity(g, cams)
        r.forward(g, cams)
        d = torch.zeros((k, sc.n, 9), device="cuda")
        r.backward(g, cams, dL.repeat(k), d_proj=d)
        torch.cuda.synchronize()
        assert r.status() == gs.GS_OK
        if k == 1:
            M = opacity_magnitudes(r, size, dL, BG)
        out.append(d[:, :, 5].double())
    one, many = out
    assert int((M > 0).sum()) > 150
    # both add the same terms: 8 in a row, 2 over rows, 8 over blocks, 49 over tiles, a division on
    # either side of the blocks; twice for a magnitude that decides a pixel at alpha_min otherwise
    bound = 2 * 2 * (8 + 2 + 8 + 49 + 2) * 2.0 ** -24 * M
    for v in range(copies):
        assert ((one[0] - many[v]).abs() <= bound).all()
