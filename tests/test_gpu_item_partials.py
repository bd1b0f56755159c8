"""Pair partials summed per item (d_proj of gs_project_bwd) in both launch forms: few and many
items (one and four runs of 32 a warp), runs longer than a window of 80 slots, ragged
last warps: equal, for the items both have, to those of the same Gaussians without
the unseen ones that make them many."""
import pytest
import torch

from paper_2506_05558_gb300 import gs, synth
from paper_2506_05558_gb300.raster import Rasterizer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


def d_proj(g, cams, sizes, dL):
    r = Rasterizer(g.n, sizes, 1 << 18, gs.config(sh_degree=0))
    r.forward(g, cams)
    assert r.status() == gs.GS_OK
    d = torch.full((g.n * len(sizes), 9), float("nan"), device="cuda")
    r.backward(g, cams, dL, d)
    torch.cuda.synchronize()
    return d.view(len(sizes), g.n, 9), r.proj.n_tiles.view(len(sizes), g.n), r.grads


@pytest.mark.parametrize("extra", [3, 311_000, 622_593])
def test_item_partials(extra):
    sizes = [(320, 200), (333, 211)]
    sc, cams, _ = synth.multiview_scene(seed=9, n=1500, n_views=2, sizes=sizes)
    g = gs.Gaussians.from_scene(sc)
    g.scale[::7] += 3.5  # splats of many tiles: runs of several windows
    cams = gs.cameras_tensor(cams)
    dL = torch.randn(3 * (320 * 200 + 333 * 211), device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    base, nt, grads = d_proj(g, cams, sizes, dL)
    assert int(nt.max()) > 80 and int((nt > 0).sum()) > 100  # the inputs hold what the test is about
    unseen = [t[:1].repeat(extra, 1) for t in (g.mean_opa, g.scale, g.quat, g.sh)]
    unseen[0][:, 2] = -1e4
    # the seen Gaussians spread over the unseen ones
    at = torch.sort(torch.randperm(1500 + extra, generator=torch.Generator().manual_seed(5))[:1500]).values.cuda()
    rows = []
    for u, t in zip(unseen, (g.mean_opa, g.scale, g.quat, g.sh)):
        a = torch.empty((1500 + extra, t.shape[1]), device="cuda")
        a[:] = u[:1]
        a[at] = t
        rows.append(a)
    got, nt2, grads2 = d_proj(gs.Gaussians(*rows), cams, sizes, dL)
    seen = nt > 0
    assert torch.equal(nt2[:, at], nt)
    assert torch.equal(got[:, at][seen], base[seen])
    assert torch.isnan(got[nt2 == 0]).all()
    assert torch.equal(grads2.scale[at], grads.scale) and torch.equal(grads2.sh[at], grads.sh)
