"""The bundle adjustment's camera solve, whose warps hand values to one another: every
number of frames (7 to 43 camera parameters: rows of up to 32 terms and of more), the
same bits from every run, and a system without positive pivots."""
import numpy as np
import pytest
import torch

from helpers import assert_close
from oracle import mini_ba as B
from paper_2506_05558_gb300 import gs
from test_gpu_ba import built, problem, run_gpu, to_device  # noqa: F401
from test_gpu_ba_sizes import clear_of_threshold

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [3, 4, 5, 6, 7, 8])
def test_cameras_of_one_iteration(F):
    for seed in range(100):
        gt, obs, cx, cy, params = problem(300 + seed, F=F, P=160)
        if clear_of_threshold(np.linalg.norm(B.residuals(params, obs, cx, cy), axis=2)):
            break
    ref, lam_ref, info = B.lm_iteration(params, 1e-5, obs, cx, cy)
    got, lam, hist = run_gpu(obs, params, 1)
    assert bool(hist[0, 2]) == info["accepted"] and abs(lam - lam_ref) < 1e-12
    # tolerances of test_one_iteration_matches_oracle
    assert abs(got["fl"] - ref["fl"]) < 1e-4 * ref["fl"]
    assert_close(got["R"], ref["R"], 1e-5, what="rotations")
    assert_close(got["t"], ref["t"], 1e-4, what="translations")


@pytest.mark.parametrize("F", [2, 6, 8])
def test_runs_agree_bit_for_bit(F):
    gt, obs, cx, cy, params = problem(7, F=F, P=500)
    first = run_gpu(obs, params, 40)
    for _ in range(5):
        again = run_gpu(obs, params, 40)
        assert first[1] == again[1] and np.array_equal(first[2], again[2], equal_nan=True)
        for k in ("fl", "R", "t", "X"):
            assert np.array_equal(np.asarray(first[0][k]), np.asarray(again[0][k]), equal_nan=True), k


def test_system_without_positive_pivots():
    """A damping of -10 makes every diagonal entry negative: the solve reports it and leaves the cameras."""
    gt, obs, cx, cy, params = problem(9, F=8, P=64)
    ob, fl, poses, pts = to_device(obs, params)
    before, f0 = poses.clone(), fl.clone()
    lam, failed = torch.tensor([-10.0], device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    gs.gs_ba_lm(ob, cx, cy, fl, poses, pts, lam, 1, gs.workspace(gs.gs_ba_workspace_size(8, 64)), failed)
    torch.cuda.synchronize()
    assert int(failed.item()) == 1
    assert torch.equal(poses, before) and torch.equal(fl, f0)  # a step of zero is exact
