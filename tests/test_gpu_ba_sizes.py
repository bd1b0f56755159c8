"""One iteration of the bundle adjustment and of the pose refinement against the
FP64 oracle at the sizes where their kernels change shape: frames from 3 to 8 (two
leave focal length and scale undetermined), points around the 16, 32 and 256 of
their chunks, one more observation a thread in the selecting cluster, and the last
size of the pose refinement's one-launch form with the first of its other form."""
import numpy as np
import pytest

from helpers import assert_close
from oracle import mini_ba as B
from test_gpu_ba import built, pose_problem, problem, run_gpu, run_pose_gpu  # noqa: F401

pytestmark = pytest.mark.gpu


def clear_of_threshold(norms):
    """No observation within FP32 reach of the rejection threshold (4 ulps)."""
    med = B.lower_median(norms)
    thr = med + 4 * B.lower_median(np.abs(norms - med))
    return np.abs(norms - thr).min() > 5e-7 * thr


@pytest.mark.parametrize("F,P", [(3, 129), (4, 33), (7, 97), (8, 31), (8, 1100)])
def test_one_iteration_at_chunk_edges(F, P):
    for seed in range(100):
        gt, obs, cx, cy, params = problem(40 + seed, F=F, P=P)
        if clear_of_threshold(np.linalg.norm(B.residuals(params, obs, cx, cy), axis=2)):
            break
    ref, lam_ref, info = B.lm_iteration(params, 1e-5, obs, cx, cy)
    got, lam, hist = run_gpu(obs, params, 1)
    assert bool(hist[0, 2]) == info["accepted"] and abs(lam - lam_ref) < 1e-12
    assert abs(hist[0, 0] - info["cost"]) < 1e-4 * info["cost"]
    assert abs(hist[0, 1] - info["trial_cost"]) < 1e-3 * info["trial_cost"]
    # tolerances of test_one_iteration_matches_oracle; of the points, all but 2%: a point whose
    # observations were mostly rejected is determined by little more than the damping floor, and
    # FP32 normal equations leave it 1e-3 off (a mistake at a chunk's edge would show in 1 of 16
    # points or more, and in the poses)
    assert abs(got["fl"] - ref["fl"]) < 1e-4 * ref["fl"]
    assert_close(got["R"], ref["R"], 1e-5, what="rotations")
    assert_close(got["t"], ref["t"], 1e-4, what="translations")
    X = ref["X"]
    off = np.abs(got["X"] - X) / (np.abs(X) + np.sqrt(np.mean(X * X)))
    assert (off.max(axis=1) > 1e-4).mean() <= 0.02 or (off.max(axis=1) > 1e-4).sum() <= 4


@pytest.mark.parametrize("M", [31, 1024, 1025, 4097, 6145, 24576, 24577])
def test_pose_iteration_at_row_edges(M):
    for seed in range(100):
        _, X, obs, cx, cy, R0, t0, _ = pose_problem(60 + seed, M=M)
        if clear_of_threshold(np.linalg.norm(B.project(500.0, cx, cy, R0, t0, X) - obs, axis=1)):
            break
    R1, t1, lam_ref, info = B.pose_lm_iteration(R0, t0, 1e-5, X, obs, 500.0, cx, cy)
    R, t, lam, hist = run_pose_gpu(X, obs, R0, t0, 1)
    assert bool(hist[0, 2]) == info["accepted"] and abs(lam - lam_ref) < 1e-12
    assert abs(hist[0, 0] - info["cost"]) < 1e-4 * info["cost"]
    # tolerances of test_pose_one_iteration_matches_oracle
    assert np.abs(R - R1).max() < 2e-6 and np.abs(t - t1).max() < 2e-6
