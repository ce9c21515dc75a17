"""Dense plans on a scene grid skip the zero columns beyond the last library
radius: results against the oracle at the edges of the skipping (odd and tiny
grids, groups cut by rows, no live column at all), and a non-finite scene or
residual value at a skipped column still makes the result NaN."""
import numpy as np
import pytest
import torch

from oracle import psfsim_oracle as O

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GRIDS = [(1, 0.5, 3.0), (7, 1.0, 2.0), (31, 0.5, 3.0), (64, 0.5, 4.0), (65, 0.3, 4.0), (90, 0.25, 2.6), (96, 0.5, 1.0),
         (12, 1.0, 0.2)]  # N, S, last radius; the last has no pixel inside


def _plan(N, S, r_last, storage, n=20, n_r=5, seed=5):
    from paper_2106_09122_gb300 import Plan
    rng = np.random.default_rng(seed)
    radii = np.linspace(0.0, r_last, n_r)
    lib = rng.uniform(0.0, 1.0, (n_r, n, n)).astype(np.float32)
    plan = Plan(torch.from_numpy(lib).to(DEV), radii, 0.25, N=N, S=S, storage=storage)
    return plan, O.build_A(lib.astype(np.float64), radii, N, S), rng


@pytest.mark.parametrize("storage,tol", [("split_bf16", 1e-5), ("bf16", 2.0 ** -8 + 2.5e-5)])
@pytest.mark.parametrize("N,S,r_last", GRIDS)
def test_forward_skips_only_zero_columns(N, S, r_last, storage, tol):
    plan, A, rng = _plan(N, S, r_last, storage)
    x = rng.uniform(0.0, 1.0, (3, N * N)).astype(np.float32)
    y = plan.forward(torch.from_numpy(x).to(DEV)).double().cpu().numpy()
    x64 = x.astype(np.float64)
    err = O.bound_relative_error(y, x64 @ A.T, x64 @ np.abs(A).T, floor=O.FLT_MIN).max()
    assert err <= tol and plan.sync_status() == 0, err


@pytest.mark.parametrize("storage", ["split_bf16", "bf16"])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_scene_value_at_a_skipped_column(storage, value):
    plan, A, rng = _plan(64, 0.5, 4.0, storage)
    dead = np.nonzero(~A.any(axis=0))[0]
    for j in (dead[0], dead[len(dead) // 2], dead[-1]):
        x = rng.uniform(0.0, 1.0, (2, 64 * 64)).astype(np.float32)
        x[1, j] = value
        y = plan.forward(torch.from_numpy(x).to(DEV)).cpu().numpy()
        assert np.isfinite(y[0]).all() and np.isnan(y[1]).all()
