"""The points at the edges of the bundle adjustment's chunks (16 and 32 points, and a last
chunk of one), one by one against the FP64 oracle after one iteration: a point alone in its
chunk moves neither poses nor a share of the points if its step is wrong. Problems are
chosen in which every such point keeps all its observations, so that it is well determined
and FP32 normal equations give it to the tolerance of the other tests."""
import numpy as np
import pytest

from oracle import mini_ba as B
from test_gpu_ba import built, problem, run_gpu  # noqa: F401
from test_gpu_ba_sizes import clear_of_threshold

pytestmark = pytest.mark.gpu


def edge_points(P):
    return sorted({i for i in (0, 15, 16, 31, 32, P - 2, P - 1) if 0 <= i < P})


@pytest.mark.parametrize("F,P", [(3, 129), (4, 33), (5, 17), (7, 97), (8, 31), (8, 33), (8, 1089)])
def test_points_at_chunk_edges(F, P):
    edges = edge_points(P)
    for seed in range(400):
        gt, obs, cx, cy, params = problem(140 + seed, F=F, P=P)
        norms = np.linalg.norm(B.residuals(params, obs, cx, cy), axis=2)
        if clear_of_threshold(norms) and B.inlier_mask(norms)[edges].all():
            break
    else:
        pytest.fail("no problem with well determined points at the edges")
    ref, _, info = B.lm_iteration(params, 1e-5, obs, cx, cy)
    got, _, hist = run_gpu(obs, params, 1)
    assert bool(hist[0, 2]) == info["accepted"]
    X = ref["X"]
    assert np.abs(X[edges] - params["X"][edges]).max(axis=1).min() > 1e-3 or not info["accepted"]  # the step is seen
    off = np.abs(got["X"][edges] - X[edges]) / (np.abs(X[edges]) + np.sqrt(np.mean(X * X)))
    assert off.max() <= 1e-4, (edges, off.max(axis=1))
