"""The focal length's right-hand side of the bundle adjustment, summed by CTAs of eight
chunks of 32 points: whole and ragged groups, chunks and a lone point at the end."""
import numpy as np
import pytest

from helpers import assert_close
from oracle import mini_ba as B
from test_gpu_ba import built, problem, run_gpu  # noqa: F401
from test_gpu_ba_sizes import clear_of_threshold

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,P", [(3, 256), (4, 257), (8, 225), (6, 289), (8, 513)])
def test_focal_step_at_group_edges(F, P):
    for seed in range(100):
        gt, obs, cx, cy, params = problem(500 + seed, F=F, P=P)
        if clear_of_threshold(np.linalg.norm(B.residuals(params, obs, cx, cy), axis=2)):
            break
    ref, lam_ref, info = B.lm_iteration(params, 1e-5, obs, cx, cy)
    got, lam, hist = run_gpu(obs, params, 1)
    assert bool(hist[0, 2]) == info["accepted"] and abs(lam - lam_ref) < 1e-12
    # tolerances of test_one_iteration_matches_oracle
    assert abs(got["fl"] - ref["fl"]) < 1e-4 * ref["fl"]
    assert_close(got["R"], ref["R"], 1e-5, what="rotations")
    assert_close(got["t"], ref["t"], 1e-4, what="translations")
