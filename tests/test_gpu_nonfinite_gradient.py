"""A pixel whose gradient is not finite, or so large that products of it overflow, reaches no
more Gaussians in a large launch (the adjoint by rows of pixels) than in a small one, and
leaves the others' gradients as they are, bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

from test_gpu_adjoint_rows import BG, gradient  # noqa: E402
from test_gpu_render_paths import run, scene  # noqa: E402

NAN, INF = float("nan"), float("inf")


@pytest.mark.parametrize("kind", ["plain", "opaque"])
@pytest.mark.parametrize("value", [NAN, INF, -INF, 3e38, 1e25])
@pytest.mark.parametrize("bg,copies,schedule", [(BG, 7, 0), ((0.0, 0.0, 0.0), 7, 1), (BG, 34, 0)])
def test_nonfinite_pixels(kind, value, bg, copies, schedule):
    size = (404, 301)
    sc, cam = scene(kind, 3000, size)
    dL = gradient(size)
    gen = torch.Generator(device="cuda").manual_seed(6)
    bad = torch.randint(0, dL.numel(), (12,), generator=gen, device="cuda")
    dL[bad] = value
    _, one = run(sc, cam, 1, schedule, dL, bg)
    _, many = run(sc, cam, copies, schedule, dL, bg)
    fine = torch.isfinite(one[0])
    if not abs(value) < INF:
        assert 0 < int((~fine[:, :6].all(1)).sum()) < sc.n // 20  # some Gaussians, not all
    for d in many:
        assert torch.isfinite(d)[fine].all()
        geometric = fine[:, :5]
        assert torch.equal(one[0, :, :5][geometric], d[:, :5][geometric])
