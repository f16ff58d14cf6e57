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


@pytest.mark.parametrize("shape,A,R", [((5,), 2, 2), ((9, 11), 3, 2), ((6, 7, 5), 4, 3), ((30, 31, 29), 3, 1),
                                       ((2, 3, 2, 3, 2), 3, 2), ((30, 30, 30, 30), 4, 4)])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("prec", [0, 1])
def test_infinities_and_nan(cp, shape, A, R, value, prec):
    """One value that is not finite. Some rows of each action's factors have a
    zero where they meet it, which makes NaN of an infinity: every state's Q is
    the value or NaN, whatever the order of the sums. A NaN of the first action
    stays, one of a later action is passed over; padding adds none of its own,
    and the residual skips NaN."""
    import torch
    dc = ci.dense_cp(shape, A, R, 0.5, seed=5)
    n = dc.nstates
    at = n // 3
    coords = np.unravel_index(at, shape)
    # where the value meets a zero of the factors (NaN), per action
    nan = np.zeros((A,) + tuple(shape), dtype=bool)
    for a in range(A):
        for r in range(R):
            for d, size in enumerate(shape):
                rows = np.arange(size) % (A + 1) == a + 1
                u = dc.factors[a][r][d]
                u[rows, coords[d]] = 0.0
                u /= u.sum(axis=1, keepdims=True)
                line = [1] * len(shape)
                line[d] = size
                nan[a] |= rows.reshape(line)
    V = ci.random_values(shape, seed=3).reshape(-1)
    V[at] = value
    q = np.where(nan, np.nan, value).reshape(A, -1)
    want, arg = q[0].copy(), np.zeros(n, dtype=np.uint8)
    with np.errstate(all="ignore"):
        for a in range(1, A):
            take = q[a] > want
            want, arg = np.where(take, q[a], want), np.where(take, a, arg)
        far = np.abs(want - V)
    f = cp.build_factors(dc, device=0)
    Vd = torch.as_tensor(V).to("cuda", torch.float64 if prec == cp.F64 else torch.float32)
    out = torch.zeros_like(Vd)
    pi = torch.full((n,), 99, dtype=torch.uint8, device="cuda")
    res = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    cp.bellman_backup(f, prec, Vd, out, pi, res)
    torch.cuda.synchronize()
    assert np.array_equal(out.double().cpu().numpy(), want, equal_nan=True)
    assert np.array_equal(pi.cpu().numpy(), arg)
    assert res.item() == (0.0 if np.isnan(far).all() else np.nanmax(far))
    f.close()
