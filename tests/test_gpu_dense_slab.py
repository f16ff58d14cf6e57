"""GPU parity of the fused mode-product chains of dense models (plans of one,
two and three phases, narrow and wide register tiles, rows cut short, values
at an odd address) against the FP64 oracle.

Tolerances as in test_gpu_dense.py: FP64 1e-12 (max|R| + max|V|); FP32
(sum_d (N_d + 2) + R + 4) 2^-24 (max|R| + max|V|).
"""
import numpy as np
import pytest

import cpmdp_inputs as ci

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24

SHAPES = [((1,), 1, 1), ((1, 1, 1), 2, 3), ((5,), 2, 2), ((2,) * 9, 3, 2), ((1, 7, 1, 9), 5, 1), ((33, 47), 3, 4),
          ((20, 21, 9), 4, 3), ((16, 17, 15, 18), 2, 3), ((30, 31, 29), 3, 1), ((300, 3), 2, 2), ((3, 301), 2, 2),
          ((130, 128, 131), 2, 1), ((40, 41, 38, 9), 3, 1), ((3000, 3), 2, 1)]


@pytest.fixture(scope="module")
def cp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build_library()
    import paper_2103_00331_gb300 as cp
    return cp


@pytest.mark.parametrize("shape,A,R", SHAPES)
@pytest.mark.parametrize("prec", [0, 1])
def test_fused_chains_one_sweep(cp, shape, A, R, prec):
    import torch
    from oracle import dense as od
    dc = ci.dense_cp(shape, A, R, 0.95, seed=5)
    n = dc.nstates
    f = cp.build_factors(dc, device=0)
    dt = torch.float64 if prec == cp.F64 else torch.float32
    buf = torch.zeros(n + 1, dtype=dt, device="cuda")
    Vd = torch.as_tensor(ci.random_values(shape, seed=1, lo=-2, hi=2).reshape(-1)).to("cuda", dt)
    Vh = Vd.double().cpu().numpy()
    Q = od.q_values(dc, Vh)
    want = Q.max(axis=0)
    scale = np.abs(dc.reward).max() + np.abs(Vh).max()
    tol = 1e-12 * scale if prec == cp.F64 else (sum(s + 2 for s in shape) + R + 4) * U32 * scale
    Qs = np.sort(Q, axis=0)
    sure = (Qs[-1] - Qs[-2]) > 2 * tol if A > 1 else np.ones(n, bool)
    first = None
    for odd in (0, 1):                      # the values at an aligned and at an odd address
        V = buf[odd:odd + n]
        V.copy_(Vd)
        out = torch.full((n,), float("nan"), dtype=dt, device="cuda")
        pi = torch.full((n,), 99, dtype=torch.uint8, device="cuda")
        res = torch.zeros(1, dtype=torch.float64, device="cuda")
        cp.bellman_backup(f, prec, V, out, pi, res)
        torch.cuda.synchronize()
        got = out.double().cpu().numpy()
        assert np.abs(got - want).max() <= tol
        assert np.array_equal(pi.cpu().numpy()[sure], Q.argmax(axis=0)[sure])
        # the residual is that of the returned values, in double
        assert res.item() == np.abs(got - Vh).max()
        if first is None:
            first = got
        else:
            assert np.array_equal(first, got)
    f.close()


@pytest.mark.parametrize("shape,A,R", [((5,), 2, 2), ((9, 11), 3, 2), ((6, 7, 5), 4, 3), ((2, 3, 2, 3, 2), 3, 1)])
def test_fused_chains_policy_iteration(cp, shape, A, R):
    """Policy iteration drives the evaluation, improvement and greedy sweeps:
    its FP64 values are the oracle's V* (to the evaluation tolerance 1e-10
    over 1 - gamma) and its policy the greedy one where the gap exceeds 1e-6."""
    import torch
    from oracle import dense as od
    dc = ci.dense_cp(shape, A, R, 0.9, seed=8)
    Vs, _, _, _ = od.value_iteration(dc, tol=1e-13, max_iter=5000)
    Q = od.q_values(dc, Vs)
    Qs = np.sort(Q, axis=0)
    sure = (Qs[-1] - Qs[-2]) > 1e-6
    f = cp.build_factors(dc, device=0)
    V = torch.zeros(dc.nstates, dtype=torch.float64, device="cuda")
    pi = torch.zeros(dc.nstates, dtype=torch.uint8, device="cuda")
    cp.policy_iteration(f, cp.F64, V, pi)
    assert np.abs(V.cpu().numpy() - Vs).max() <= 2e-9
    assert np.array_equal(pi.cpu().numpy()[sure], Q.argmax(axis=0)[sure])
    f.close()
