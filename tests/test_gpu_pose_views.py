"""gs_pose_apply and gs_pose_tangent_grad, a warp per view: every view's result is that of a
call for the view alone, for one view and the most, in place too, at angles on both sides
of the series' limit (1e-3)."""
import numpy as np
import pytest
import torch

from paper_2506_05558_gb300 import gs, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


@pytest.mark.parametrize("nv", [1, 5, 64])
@pytest.mark.parametrize("size", [0.0, 3e-4, 1.0])
def test_views_match_single_calls(nv, size):
    rng = np.random.default_rng(nv)
    cams = gs.cameras_tensor([synth.camera(np.linalg.qr(rng.standard_normal((3, 3)))[0], rng.standard_normal(3),
                                           400.0 + k, 640 + k, 480) for k in range(nv)])
    gen = torch.Generator("cuda").manual_seed(nv)
    xi = size * torch.randn((nv, 6), device="cuda", generator=gen)
    d = torch.randn((nv, 6), device="cuda", generator=gen)
    out, grad = torch.zeros_like(cams), torch.zeros_like(d)
    gs.gs_pose_apply(cams, xi, nv, out)
    gs.gs_pose_tangent_grad(xi, d, nv, grad)
    rows, outs = cams.view(nv, -1), out.view(nv, -1)
    for k in range(nv):
        one, g = torch.zeros_like(rows[k]), torch.zeros((1, 6), device="cuda")
        gs.gs_pose_apply(rows[k].contiguous(), xi[k:k + 1].contiguous(), 1, one)
        gs.gs_pose_tangent_grad(xi[k:k + 1].contiguous(), d[k:k + 1].contiguous(), 1, g)
        assert torch.equal(one, outs[k]) and torch.equal(g[0], grad[k])
    place = cams.clone()
    gs.gs_pose_apply(place, xi, nv, place)
    assert torch.equal(place, out)
    if size == 0.0:
        assert torch.equal(out, cams) and torch.equal(grad, d)
