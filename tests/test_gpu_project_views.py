"""gs_project with its CTAs' views split or not (few or many Gaussians) and ragged last
blocks: every view's rows are those of a call for that view alone, bit for bit."""
import pytest
import torch

from paper_2506_05558_gb300 import gs, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n,views,f3d", [(1, 1, False), (31, 5, True), (129, 20, False), (4099, 3, True),
                                         (480_001, 2, False)])
def test_views_match_single_calls(n, views, f3d, deg):
    sizes = [(320, 180), (200, 333), (64, 64)]
    sizes = [sizes[v % 3] for v in range(views)]
    sc, cams, _ = synth.multiview_scene(seed=n + deg, n=min(n, 4099), n_views=views, sizes=sizes)
    g = gs.Gaussians.from_scene(sc)
    if n > 4099:  # the scene's rows again, moved a little
        k = -(-n // 4099)
        rep = [t.repeat(k, 1)[:n].contiguous() for t in (g.mean_opa, g.scale, g.quat, g.sh)]
        rep[0][:, :3] += 0.5 * torch.randn((n, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        g = gs.Gaussians(*rep)
    g.sh.copy_(0.3 * torch.randn(g.sh.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(2)))
    if f3d:
        g.filter3d = 1e-3 * torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    cfg = gs.config(sh_degree=deg, mip_filter=int(f3d))
    out = gs.Projected.alloc(n * views)
    gs.gs_project(g, gs.cameras_tensor(cams), gs.frame(sizes), cfg, out)
    listed = 0
    for v in range(views):
        one = gs.Projected.alloc(n)
        gs.gs_project(g, gs.cameras_tensor(cams[v:v + 1]), gs.frame(sizes[v:v + 1]), cfg, one)
        listed += int((one.n_tiles > 0).sum())
        for k in ("mean2d", "conic_opa", "rgb_depth", "rect", "n_tiles"):
            a, b = getattr(out, k)[v * n:(v + 1) * n], getattr(one, k)
            assert torch.equal(a, b), (k, v)
    assert n < 100 or listed > 0
