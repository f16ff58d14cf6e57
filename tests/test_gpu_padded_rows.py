"""FP32 solves of grids whose rows are no multiple of 4 states (solved on
padded rows) against the grid-barrier solver on the rows as they are
(fused = 2): the same values, policies, sweep counts, residuals and counted
backups, bit for bit; a solve after another, from another start, too."""
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


@pytest.mark.parametrize("shape", [(301,), (1023,), (90, 3), (17, 19), (50, 6), (300, 301), (7, 9, 11), (31, 29, 33),
                                   (2, 3, 63), (40, 1, 7), (101, 97, 103), (5, 6, 7, 9), (130, 2)])
@pytest.mark.parametrize("kind", ["vi", "pi"])
def test_padded_rows_equal_grid_barrier(cp, shape, kind):
    import torch
    gw = ci.gridworld(shape, p=0.8, gamma=0.93, step_reward=-0.04, goal_rewards=[1.0, -1.0], obstacle_rate=0.1, seed=4)
    n = gw.nstates
    f = cp.build_factors(gw, device=0)
    solve = cp.value_iteration if kind == "vi" else cp.policy_iteration
    starts = [torch.zeros(n, dtype=torch.float32, device="cuda"),
              torch.as_tensor(ci.random_values(shape, seed=2).reshape(-1).astype(np.float32)).cuda()]
    buf = torch.zeros(n + 1, dtype=torch.float32, device="cuda")
    for start in starts:
        got = []
        for fused, V in ((2, start.clone()), (1, start.clone()), (1, buf[1:].copy_(start))):   # and an odd address
            pi = torch.full((n,), 77, dtype=torch.uint8, device="cuda")
            r = solve(f, cp.F32, V, pi, opts=cp.default_opts(fused=fused, max_iter=400), raise_on_noconv=False)
            got.append((V.cpu().numpy().copy(), pi.cpu().numpy(), r))
        for V, pi, r in got[1:]:
            assert np.array_equal(V, got[0][0])
            assert np.array_equal(pi, got[0][1])
            for k in ("status", "iterations", "rounds", "eval_sweeps", "residual", "certified_residual", "backups"):
                assert r[k] == got[0][2][k], k
    f.close()


def test_padded_rows_trace_and_limit(cp):
    """The residual trace and a solve that reaches its sweep limit."""
    import torch
    gw = ci.gridworld((33, 35), p=0.8, gamma=0.99, step_reward=-0.04, goal_rewards=[1.0], obstacle_rate=0.05, seed=6)
    f = cp.build_factors(gw, device=0)
    out = []
    for fused in (2, 1):
        V = torch.zeros(gw.nstates, dtype=torch.float32, device="cuda")
        tr = torch.full((20,), -1.0, dtype=torch.float64, device="cuda")
        r = cp.value_iteration(f, cp.F32, V, None, opts=cp.default_opts(fused=fused, max_iter=20, certify=0, trace=tr.data_ptr()),
                               raise_on_noconv=False)
        out.append((V.cpu().numpy(), tr.cpu().numpy(), r["iterations"], r["status"], r["residual"]))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][2:] == out[1][2:] and out[0][3] == cp.ENOCONV
    assert np.array_equal(out[0][1], out[1][1])
    f.close()
