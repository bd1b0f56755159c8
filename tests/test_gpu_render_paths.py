"""The compositing kernels of large launches against those of small ones.

A view of 494 tiles takes the one-pixel-per-thread kernels; four copies of it in
one launch (1,976 tiles) take the 8x8-block forward and the row adjoint. Both
must give each copy the same image, transmittance and contributor count bit for
bit, and the same projected gradients: the geometric ones bit for bit, the colour
and opacity sums up to the order of their additions."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2506_05558_gb300 import gs, synth  # noqa: E402
from paper_2506_05558_gb300.raster import Rasterizer  # noqa: E402


def scene(kind, n, size):
    sc, cams, rng = synth.multiview_scene(seed=31, n=n, n_views=1, sizes=[size])
    if kind == "opaque":  # alpha reaches alpha_max, pixels terminate early
        sc.mean_opa[:, 3] = rng.normal(4.0, 4.0, n)
        sc.scale[:, :3] += 1.0
    elif kind == "thin":  # needles of up to hundreds of pixels, too thin for the exact block test
        sc.scale[: n // 2, 0] += 4.0
        sc.scale[: n // 2, 1:3] -= 4.0
    elif kind == "large":  # every entry touches all blocks of its tiles
        sc.scale[:, :3] += 3.0
    return sc, cams[0]


def run(sc, cam, copies, schedule, dL, background):
    w, h = cam["width"], cam["height"]
    cfg = gs.config(sh_degree=3, schedule=schedule, bg=background)
    r = Rasterizer(sc.n, [(w, h)] * copies, 1 << 16, cfg)
    r.img.depth = torch.zeros_like(r.img.t_final)
    g, cams = gs.Gaussians.from_scene(sc), gs.cameras_tensor([cam] * copies)
    r.fit_capacity(g, cams)
    r.forward(g, cams)
    d_proj = torch.zeros((copies, sc.n, 9), device="cuda")
    r.backward(g, cams, dL.repeat(copies), d_proj=d_proj)
    torch.cuda.synchronize()
    assert r.status() == gs.GS_OK
    img = r.img
    return [t.view(copies, -1) for t in (img.color, img.t_final, img.n_contrib, img.depth)], d_proj


@pytest.mark.parametrize("kind,n,size,schedule", [
    ("plain", 6000, (403, 301), 0), ("plain", 6000, (404, 304), 1), ("opaque", 20000, (403, 301), 2),
    ("opaque", 3, (403, 301), 0), ("thin", 4000, (403, 301), 0), ("large", 3000, (404, 303), 0)])
def test_large_launch_matches_small(kind, n, size, schedule):
    sc, cam = scene(kind, n, size)
    w, h = size
    gen = torch.Generator(device="cuda").manual_seed(5)
    dL = torch.randn(3 * w * h, generator=gen, device="cuda")
    bg = (0.3, 0.1, 0.7)
    one, d_one = run(sc, cam, 1, schedule, dL, bg)
    many, d_many = run(sc, cam, 4, schedule, dL, bg)
    _, d_abs = run(sc, cam, 1, schedule, dL.abs(), bg)  # sums of the colour terms' magnitudes
    for a, b in zip(one, many):
        for v in range(4):
            assert torch.equal(a[0], b[v])
    # additions a colour or opacity term passes through: 8 in a row, 3 over rows and halves, 8 over
    # blocks and one per tile of its Gaussian (at most 494); each rounds by 2^-24 of the partial sum
    steps = 19 + 494
    for v in range(4):
        assert torch.equal(d_one[0, :, :5], d_many[v, :, :5])
        colour = (d_one[0, :, 6:] - d_many[v, :, 6:]).abs()
        assert (colour <= 2 * steps * 2.0 ** -24 * d_abs[0, :, 6:]).all()
        o, p = d_one[0, :, 5].double(), d_many[v, :, 5].double()
        assert (o - p).abs().max() <= 2 * steps * 2.0 ** -24 * float(o.abs().max()) * 8 + 1e-30
