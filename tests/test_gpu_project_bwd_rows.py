"""Rows of gs_project_bwd wherever a Gaussian lies in its CTA's blocks: unseen Gaussians put in
front shift every row and change nothing but that (bit for bit), theirs are zero, and
accumulate adds to what is there."""
import pytest
import torch

from paper_2506_05558_gb300 import gs, synth
from paper_2506_05558_gb300.raster import Rasterizer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


def grads(g, cams, sizes, cfg, dL, fill):
    r = Rasterizer(g.n, sizes, 1 << 16, cfg)
    for t, f in zip((r.grads.mean_opa, r.grads.scale, r.grads.quat, r.grads.sh), fill):
        t.copy_(f)
    r.forward(g, cams)
    assert r.status() == gs.GS_OK
    r.backward(g, cams, dL)
    torch.cuda.synchronize()
    return [r.grads.mean_opa, r.grads.scale, r.grads.quat, r.grads.sh, r.grads.visible]


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n,views,front,accumulate", [(1, 1, 31, 0), (97, 2, 1, 1), (300, 3, 127, 0), (300, 17, 5, 1),
                                                      (513, 16, 130, 1)])
def test_rows_shift(n, views, front, accumulate, deg):
    sizes = [(96, 64)] * views
    sc, cams, _ = synth.multiview_scene(seed=n + deg, n=n, n_views=views, sizes=sizes)
    gen = torch.Generator("cuda").manual_seed(7)
    g = gs.Gaussians.from_scene(sc)
    g.sh.copy_(0.3 * torch.randn(g.sh.shape, device="cuda", generator=gen))
    g.scale += 1.5  # some splats of several tiles
    unseen = gs.Gaussians(*[t[:1].repeat(front, 1) for t in (g.mean_opa, g.scale, g.quat, g.sh)])
    unseen.mean_opa[:, 2] = -1e4
    both = gs.Gaussians(*[torch.cat([getattr(unseen, k), getattr(g, k)]).contiguous()
                          for k in ("mean_opa", "scale", "quat", "sh")])
    cams = gs.cameras_tensor(cams)
    dL = torch.randn(3 * 96 * 64 * views, device="cuda", generator=gen)
    fill = [torch.randn(t.shape, device="cuda", generator=gen) for t in (both.mean_opa, both.scale, both.quat, both.sh)]
    base = grads(g, cams, sizes, gs.config(sh_degree=deg), dL, [f[front:] for f in fill])
    got = grads(both, cams, sizes, gs.config(sh_degree=deg, accumulate=accumulate), dL, fill)
    assert n == 1 or int(base[4].sum()) > 0
    for a, b, f in zip(got[:4], base[:4], fill):
        old = f if accumulate else torch.zeros_like(f)
        assert torch.equal(a[:front], old[:front])
        assert torch.equal(a[front:], b + old[front:])
    assert not got[4][:front].any() and torch.equal(got[4][front:], base[4])
