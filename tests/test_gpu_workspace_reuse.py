"""Calls in a workspace that was sized for a larger one give what they give in their own."""
import numpy as np
import pytest
import torch

from paper_2506_05558_gb300 import gs, synth
from paper_2506_05558_gb300.raster import Rasterizer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


def poisoned(size):
    ws = gs.workspace(size)
    ws.view(torch.uint8).fill_(0xA5)
    return ws


def test_sort_below_the_edge_of_its_radix_tiles():
    sc, cams, _ = synth.multiview_scene(seed=51, n=6000, n_views=1, sizes=[(640, 480)])
    g, cam = gs.Gaussians.from_scene(sc), gs.cameras_tensor(cams)
    r = Rasterizer(g.n, [(640, 480)], 1 << 20)
    gs.gs_project(g, cam, r.f, r.cfg, r.proj)
    larger = gs.gs_sort_workspace_size(g.n, r.f, (1 << 20) + 1)
    lists = []
    for ws in (r.ws_sort, poisoned(larger)):
        gs.gs_sort(r.proj, g.n, r.f, r.pairs, ws)
        torch.cuda.synchronize()
        assert r.status() == gs.GS_OK
        lists.append((r.pairs.range.clone(), r.pairs.src[:r.pair_count()].clone(), r.pairs.emit[:r.pair_count()].clone()))
    assert lists[0][1].numel() > 0
    for a, b in zip(*lists):
        assert torch.equal(a, b)


def spawn(kind, W, H, ws):
    gen = torch.Generator(device="cuda").manual_seed(W)
    image = torch.rand((3, H, W), generator=gen, device="cuda")
    depth = 1 + torch.rand((H, W), generator=gen, device="cuda")
    cam = gs.cameras_tensor([synth.camera(np.eye(3), np.zeros(3), 100.0, W, H)])
    out = gs.Spawned.alloc(W * H)
    if kind == "propose":
        gs.gs_spawn_propose(image, None, depth, W, H, cam, 1.0, 5, 1, out, ws)
    else:
        mlp_out = torch.randn((gs.gs_mlp_patches(W, H), 3), generator=gen, device="cuda")
        gs.gs_spawn_learned(image, mlp_out, W, H, cam, 5, 1, out, ws, depth=depth)
    torch.cuda.synchronize()
    n = int(out.count.item())
    assert n > 0 and int(out.status.item()) == gs.GS_OK
    return [t[:n].clone() for t in (out.g.mean_opa, out.g.scale, out.g.sh)]


# the second shapes have more mask words (one per 32 pixels of a row) than the workspace's frame
@pytest.mark.parametrize("kind,sized,shape", [("learned", (1920, 1080), (1080, 1920)), ("learned", (640, 40), (40, 640)),
                                              ("propose", (640, 40), (1, 25600)), ("propose", (64, 64), (2, 2048))])
def test_spawn_of_another_shape(kind, sized, shape):
    ws = poisoned(gs.gs_spawn_workspace_size(*sized))
    own = poisoned(gs.gs_spawn_workspace_size(*shape))
    for a, b in zip(spawn(kind, *shape, own), spawn(kind, *shape, ws)):
        assert torch.equal(a, b)
