"""Fused mode-product chains of dense models on values at the ends of the
floating-point range, in both register tiles of the last run of modes."""
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


@pytest.mark.parametrize("shape,A,R", [((5,), 2, 2), ((9, 11), 3, 2), ((30, 30, 30, 30), 4, 4)])
def test_residual_past_the_largest_float(cp, shape, A, R):
    """Values of -3e38 and rewards up to 3e38: V' - V overflows a float in some
    states, not in others; the residual is the largest difference, in double."""
    import torch
    dc = ci.dense_cp(shape, A, R, 0.1, seed=5)
    n = dc.nstates
    dc.reward[...] = (3e38 * ci.uniform(7, 1, n)).reshape(shape)
    dc.reward.reshape(-1)[n // 2] = 3e38
    f = cp.build_factors(dc, device=0)
    V = torch.full((n,), -3e38, dtype=torch.float32, device="cuda")
    out = torch.empty_like(V)
    res = torch.zeros(1, dtype=torch.float64, device="cuda")
    cp.bellman_backup(f, cp.F32, V, out, None, res)
    torch.cuda.synchronize()
    far = (out.double() - V.double()).abs().max().item()
    assert np.isfinite(far) and far > 4e38
    assert res.item() == far
    f.close()
