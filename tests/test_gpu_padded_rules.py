"""Which solver a grid of ragged rows takes, on padded rows or as it is, and
that its results are those of the grid barrier on the rows as they are
(fused = 2): solves of few sweeps, policy iteration of more states than
columns of two segments hold, value iteration of 2^23 states and more."""
import numpy as np
import pytest

import cpmdp_inputs as ci

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build_library()
    import paper_2103_00331_gb300 as cp
    return cp


@pytest.mark.parametrize("shape,kind,limit,solver", [
    ((33, 35), "vi", 11, "GRID_BARRIER"), ((33, 35), "vi", 12, "BARRIER_FREE"), ((33, 35), "pi", 3, "GRID_BARRIER"),
    ((33, 35), "pi", 4, "BARRIER_FREE"), ((75, 73, 74), "vi", 30, "BARRIER_FREE"), ((75, 73, 74), "pi", 6, "GRID_BARRIER"),
    ((65, 66, 63), "pi", 6, "BARRIER_FREE"), ((99, 101, 103), "vi", 2, "GRID_BARRIER"),
    ((203, 207, 205), "vi", 13, "GRID_BARRIER"), ((203, 207, 205), "pi", 4, "GRID_BARRIER")])
def test_solver_and_results(cp, shape, kind, limit, solver):
    import torch
    gw = ci.gridworld(shape, p=0.8, gamma=0.93, step_reward=-0.04, goal_rewards=[1.0, -1.0], obstacle_rate=0.1, seed=4)
    f = cp.build_factors(gw, device=0)
    solve = cp.value_iteration if kind == "vi" else cp.policy_iteration
    got = []
    for fused in (2, 1):
        V = torch.zeros(gw.nstates, dtype=torch.float32, device="cuda")
        pi = torch.full((gw.nstates,), 77, dtype=torch.uint8, device="cuda")
        r = solve(f, cp.F32, V, pi, opts=cp.default_opts(fused=fused, max_iter=limit, max_rounds=limit), raise_on_noconv=False)
        got.append((V.cpu().numpy(), pi.cpu().numpy(), r))
    assert got[1][2]["solver"] == getattr(cp, "SOLVER_" + solver)
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    for k in ("status", "iterations", "rounds", "eval_sweeps", "residual", "certified_residual", "backups"):
        assert got[0][2][k] == got[1][2][k], k
    f.close()
