"""The Function's pair buffer: a hint that is too small, exact or ample, an empty view
and accumulate = 1 give the raw calls' image and gradients, bit for bit (the same
kernels on buffers that are not zero-filled)."""
import pytest
import torch

from paper_2506_05558_gb300 import gs, synth
from paper_2506_05558_gb300.autograd import rasterize
from paper_2506_05558_gb300.raster import Rasterizer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


@pytest.mark.parametrize("accumulate", [0, 1])
@pytest.mark.parametrize("hint", [1, "exact", 1 << 20])
@pytest.mark.parametrize("away", [False, True])
def test_fit(hint, away, accumulate):
    sc, cam, _ = synth.tiny_scene()
    sizes = [(64, 64), (64, 64)]
    cams = [cam, cam]
    if away:  # the second camera looks at nothing
        cams = [cam, dict(cam, t=cam["t"] - [0.0, 0.0, 1e4])]
    cams = gs.cameras_tensor(cams)
    cfg = gs.config(sh_degree=0, bg=(0.2, 0.1, 0.0), accumulate=accumulate)
    g = gs.Gaussians.from_scene(sc)
    dL = torch.randn(2 * 3 * 64 * 64, generator=torch.Generator().manual_seed(3)).cuda()
    xi = torch.zeros((2, 6), device="cuda")
    applied = torch.empty_like(cams)
    gs.gs_pose_apply(cams, xi, 2, applied)
    r = Rasterizer(sc.n, sizes, 1 << 16, cfg)
    pairs = r.fit_capacity(g, applied)
    r.forward(g, applied)
    r.backward(g, applied, dL)
    d_xi = torch.empty_like(r.dpose)
    gs.gs_pose_tangent_grad(xi, r.dpose, 2, d_xi)
    # blocks with other contents for the Function's buffers to land in
    junk = [torch.full((k,), float("nan"), device="cuda") for k in (1000, 10_000, 100_000, 1_000_000, 3_000_000)]
    del junk
    leaves = [t.clone().requires_grad_(True) for t in (g.mean_opa, g.scale, g.quat, g.sh, xi)]
    color, t_final = rasterize(*leaves, cams, sizes, cfg, pairs if hint == "exact" else hint)
    grads = torch.autograd.grad(color, leaves, dL)
    assert torch.equal(color, r.img.color) and torch.equal(t_final, r.img.t_final)
    for got, want in zip(grads, (r.grads.mean_opa, r.grads.scale, r.grads.quat, r.grads.sh, d_xi)):
        assert torch.equal(got, want)
