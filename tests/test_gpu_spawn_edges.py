"""Spawn proposal at the edges of its launches (tiles of 64 x 16 pixels, threads of
4 x 2, mask words of 32, warps of 8 words): ragged and narrow frames, every tap
radius, a depth map that is not 16-byte aligned, no maps, a cut capacity, and the
largest narrow frame of the call without scratch. Tolerance of a map value: the
rounding bound of a sum of n taps of values in [0, 1] over three channels,
sqrt(3) (n + 2) 2^-24 sum |w|; the mask may differ where u is that near to P_s."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2506_05558_gb300 import gs, synth
from test_gpu_spawn import smooth_image, t32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    from oracle import build as ob
    build.build()
    ob.build()


def map_bound(sigma):
    R = int(np.ceil(3 * sigma))
    j, i = np.mgrid[-R:R + 1, -R:R + 1]
    r2, s2 = i * i + j * j, sigma * sigma
    w = (r2 - 2 * s2) / s2 ** 2 * np.exp(-r2 / (2 * s2)) / (2 * np.pi * s2)
    w -= w.mean()
    return np.sqrt(3) * (w.size + 2) * 2.0 ** -24 * np.abs(w).sum()


def proposal(im, rd, depth, W, H, cam, sigma, seed, frame, cap, maps=True):
    out = gs.Spawned.alloc(cap, W * H) if maps else gs.Spawned.alloc(cap)
    ws = gs.workspace(gs.gs_spawn_workspace_size(W, H))
    ws.view(torch.uint8).fill_(0xA5)  # nothing in it may have to start at zero
    gs.gs_spawn_propose(im, rd, depth, W, H, cam, sigma, seed, frame, out, ws, capacity=cap)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("sigma", [0.3, 0.6, 1.0, 1.3, 1.6, 2.0, 2.3, 8 / 3])
@pytest.mark.parametrize("W,H,render,shift", [(1, 41, True, 0), (2, 3, False, 0), (31, 17, True, 0), (33, 5, False, 1),
                                              (64, 16, True, 0), (68, 33, True, 1), (130, 47, True, 0)])
def test_spawn_edges(W, H, render, shift, sigma):
    rng = np.random.default_rng(W + H)
    im = smooth_image(rng, W, H)
    rd = np.clip(im + 0.3 * rng.standard_normal(im.shape), 0, 1).astype(np.float32) if render else None
    depth = rng.uniform(1.0, 20.0, (H, W)).astype(np.float32)
    depth[::3, ::5] = 0.0
    depth[1::7, ::4] = np.inf
    z = torch.zeros(W * H + shift, device="cuda")
    z[shift:] = t32(depth).reshape(-1)
    cam = synth.camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 0.8 * W, W, H)
    cams, img = gs.cameras_tensor([cam]), t32(im)
    rnd = None if rd is None else t32(rd)
    out = proposal(img, rnd, z[shift:], W, H, cams, sigma, 7, 2, W * H)
    n = int(out.count.item())
    assert int(out.status.item()) == gs.GS_OK
    tol = map_bound(sigma)
    ref = O.spawn(im.astype(np.float64), None if rd is None else rd.astype(np.float64), depth, cam, sigma, 7, 2,
                  margin=2 * tol + 2.0 ** -24)
    m = ref["maps"]
    for k, f in (("p_l", 1), ("p_pen", 1), ("p_s", 2)):
        err = np.abs(getattr(out, k).cpu().numpy().reshape(H, W) - m[k]).max()
        assert err <= f * tol + 2.0 ** -23, (k, err, tol)
    pix = out.pixel[:n].cpu().numpy()
    assert np.all(np.diff(pix) > 0)
    amb = set(np.nonzero(m["amb"].reshape(-1))[0].tolist())
    assert (set(pix.tolist()) ^ set(ref["pixel"].tolist())) <= amb
    # rows from the values that the maps hold: nearest-neighbour scale, colour, depth along the ray
    pl = out.p_l.double().cpu().numpy().reshape(-1)[pix]
    d = depth.reshape(-1)[pix].astype(np.float64)
    mo, sc = out.g.mean_opa[:n].double().cpu().numpy(), out.g.scale[:n].double().cpu().numpy()
    assert np.all(mo[:, 2] == d) and np.all(mo[:, 3] == 0)
    want = np.log(d * 0.5 / np.sqrt(pl) / float(np.float32(0.8 * W)))
    assert np.all(np.abs(sc[:, :3] - want[:, None]) <= 2.0 ** -20 + 2.0 ** -22 * np.abs(want[:, None]))
    assert np.all(out.g.quat[:n].cpu().numpy() == np.array([1, 0, 0, 0], np.float32))
    sh = out.g.sh[:n].double().cpu().numpy().reshape(n, 48)
    dc = (im.reshape(3, -1).T[pix].astype(np.float64) - 0.5) * 2 * np.sqrt(np.pi)
    assert np.all(np.abs(sh[:, :3] - dc) <= 2.0 ** -21) and not sh[:, 3:].any()
    # without maps, and with room for some of the spawns: the same rows
    for cap in (W * H, max(n // 2, 1), 0):
        o2 = proposal(img, rnd, z[shift:], W, H, cams, sigma, 7, 2, cap, maps=False)
        assert int(o2.count.item()) == n
        assert int(o2.status.item()) == (gs.GS_ERR_CAPACITY if n > cap else gs.GS_OK)
        k = min(n, cap)
        for a, b in ((o2.g.mean_opa, out.g.mean_opa), (o2.g.scale, out.g.scale), (o2.g.quat, out.g.quat),
                     (o2.g.sh, out.g.sh)):
            assert torch.equal(a[:k], b[:k])


@pytest.mark.parametrize("W,H", [(2, 65535 * 16), (1 << 21, 1), (33, 63550)])
def test_noalloc_largest_frames(W, H):
    g = torch.Generator().manual_seed(1)
    im = torch.rand(3, H, W, generator=g).cuda()
    depth = torch.rand(H, W, generator=g).cuda() + 1
    cams = gs.cameras_tensor([synth.camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), 50.0, W, H)])
    a = proposal(im, None, depth, W, H, cams, 1.0, 3, 1, 1000, maps=False)
    b = gs.Spawned.alloc(1000)
    gs.gs_spawn_propose_noalloc(im, None, depth, W, H, cams, 1.0, 3, 1, b)
    torch.cuda.synchronize()
    assert int(a.count.item()) == int(b.count.item()) > 1000
    assert int(a.status.item()) == int(b.status.item()) == gs.GS_ERR_CAPACITY
    for x, y in ((a.g.mean_opa, b.g.mean_opa), (a.g.scale, b.g.scale), (a.g.sh, b.g.sh)):
        assert torch.equal(x, y)
