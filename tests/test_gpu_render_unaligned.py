"""Buffers that start anywhere on a float: the adjoint of large launches reads rows of
eight pixels 16 bytes at a time where it may, and gives the same bits where the image or
the gradient is a slice that it may not read so."""
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2506_05558_gb300 import gs, synth  # noqa: E402
from paper_2506_05558_gb300.autograd import rasterize  # noqa: E402
from paper_2506_05558_gb300.raster import Rasterizer  # noqa: E402

W, H, COPIES = 404, 304, 4  # 1,976 tiles; widths and views in whole 16 bytes


def scene():
    sc, cams, _ = synth.multiview_scene(seed=37, n=6000, n_views=1, sizes=[(W, H)])
    return gs.Gaussians.from_scene(sc), gs.cameras_tensor([cams[0]] * COPIES)


def offset(t, k):
    """A copy of t that starts k elements into its buffer."""
    buf = torch.empty((t.numel() + k,), dtype=t.dtype, device=t.device)
    buf[k:] = t
    return buf[k:]


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("which", ["t_final", "n_contrib", "gradient"])
def test_offset_buffer_gives_the_same_bits(which, k):
    g, cams = scene()
    r = Rasterizer(g.n, [(W, H)] * COPIES, 1 << 18)
    r.fit_capacity(g, cams)
    r.forward(g, cams)
    gen = torch.Generator(device="cuda").manual_seed(3)
    dL = torch.randn(r.img.color.shape, generator=gen, device="cuda")
    want, got = (torch.zeros((COPIES, g.n, 9), device="cuda") for _ in range(2))
    r.backward(g, cams, dL, d_proj=want)
    if which == "gradient":
        dL = offset(dL, k)
        assert dL.data_ptr() % 16 == 4 * k
    else:
        setattr(r.img, which, offset(getattr(r.img, which), k))
    r.backward(g, cams, dL, d_proj=got)
    torch.cuda.synchronize()
    assert r.status() == gs.GS_OK and float(want.abs().max()) > 0
    assert torch.equal(want, got)


def test_gradient_behind_another_render():
    """torch.cat's backward hands each render a slice of one gradient."""
    g, cams = scene()
    small = (33, 17)  # 1,683 values: what follows them is not on 16 bytes
    cam_small = gs.cameras_tensor(synth.multiview_scene(seed=38, n=10, n_views=1, sizes=[small])[1])
    gen = torch.Generator(device="cuda").manual_seed(4)
    weight = torch.randn(3 * (small[0] * small[1] + COPIES * W * H), generator=gen, device="cuda")

    starts = []

    def grads(both):
        leaves = [t.clone().requires_grad_(True) for t in (g.mean_opa, g.scale, g.quat, g.sh)]
        xi = torch.zeros((COPIES, 6), device="cuda", requires_grad=True)
        color, _ = rasterize(*leaves, xi, cams, [(W, H)] * COPIES)
        if both:
            first, _ = rasterize(*(t.detach() for t in leaves), torch.zeros((1, 6), device="cuda"), cam_small, [small])
            color.register_hook(lambda d: starts.append(d.data_ptr() % 16))
            color = torch.cat([first, color])
        (color * weight[-color.numel():]).sum().backward()
        return [t.grad for t in (*leaves, xi)]

    for a, b in zip(grads(False), grads(True)):
        assert torch.equal(a, b)
    assert starts[0] != 0
