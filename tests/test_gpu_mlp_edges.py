"""The fused training step (tcgen05) at the edges of its launches: splits of 256 patches in
tiles of 128, sums over more than 36 splits, a workspace of NaNs, gradients or Adam alone.
Loss and gradients against the oracle with the bounds of the whole step's test, and
outputs and gradients against the product chain (an image off 16-byte alignment takes
it): the same products in the same order, where one activation's rounding to bfloat16
may differ by 2^-8 of itself."""
import numpy as np
import pytest
import torch

from helpers import assert_close
from paper_2506_05558_gb300 import gs
from test_gpu_mlp import mlp_case, oracle_train

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2506_05558_gb300 import build
    build.build()


def train(layers, image, targets, shift=0, want_grads=True, adam=True):
    H, W = image.shape[1:]
    n = gs.gs_mlp_patches(W, H)
    p = gs.MlpParams.from_numpy(layers)
    m, v = (gs.MlpParams.zeros(), gs.MlpParams.zeros()) if adam else (None, None)
    ws = gs.workspace(gs.gs_mlp_workspace_size(n))
    ws.fill_(0xFF)
    loss, out = torch.zeros(1, device="cuda"), torch.zeros((n, 3), device="cuda")
    grads = torch.zeros(gs.gs_mlp_param_count(), device="cuda") if want_grads else None
    buf = torch.zeros(image.size + shift, device="cuda")
    buf[shift:] = torch.tensor(image, dtype=torch.float32, device="cuda").reshape(-1)
    tg = torch.tensor(targets, dtype=torch.float32, device="cuda")
    gs.gs_mlp_train_step(p, m, v, buf[shift:], W, H, tg, gs.mlp_config(tensor_path=1, lr=1e-3), 1, loss, ws, out=out,
                         grads=grads)
    torch.cuda.synchronize()
    assert gs.gs_mlp_tc_error() == 0
    flat = np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in p.numpy()])
    return loss.item(), out.cpu().numpy(), None if grads is None else grads.cpu().numpy(), flat


@pytest.mark.parametrize("W,H", [(8, 8), (8 * 43, 24), (128, 128), (8 * 257, 8), (8 * 97, 8 * 96)])
def test_train_step_edges(W, H):
    rng, layers, image, targets = mlp_case(W + H, W=W, H=H)
    loss, out, grads, params = train(layers, image, targets)
    _, L, g, _ = oracle_train(layers, image, targets)
    assert abs(loss - L) <= 1e-3 * abs(L)
    off = 0
    for l, (dW, db) in enumerate(g):
        for name, ref in ((f"dW{l + 1}", dW), (f"db{l + 1}", db)):
            assert_close(grads[off:off + ref.size].reshape(ref.shape), ref, 1e-2, what=name)
            off += ref.size
    loss_c, out_c, grads_c, _ = train(layers, image, targets, shift=1)
    assert abs(loss - loss_c) <= 1e-5 * abs(loss_c) and np.abs(out - out_c).max() <= 2.0 ** -8 * np.abs(out_c).max()
    assert np.linalg.norm(grads - grads_c) <= 2.0 ** -8 * np.linalg.norm(grads_c)
    # gradients alone leave the parameters, Adam alone takes the same step
    loss_g, _, grads_g, params_g = train(layers, image, targets, adam=False)
    assert loss_g == loss and np.array_equal(grads_g, grads)
    assert np.array_equal(params_g, np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in layers])
                          .astype(np.float32))
    assert np.array_equal(train(layers, image, targets, want_grads=False)[3], params)
