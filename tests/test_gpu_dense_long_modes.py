"""Dense sweeps with modes of about 1,024 states and more, by the fused chains or
by one launch per mode, against the same products in FP64. Rows of the factors
sum to 1, so each of an output's N additions rounds at most max|V|: N 2^-24
(FP64: 2^-53) of it per mode, and as much again for the sum over ranks, R and
gamma."""
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


@pytest.mark.parametrize("shape,A,R", [((1024,), 2, 1), ((1025,), 2, 1), ((1400,), 2, 2), ((1400,), 4, 4), ((1300, 3), 2, 1),
                                       ((2, 1300), 2, 1), ((1300, 32), 2, 2), ((2050,), 1, 1)])
@pytest.mark.parametrize("prec", ["F32", "F64"])
def test_sweep(cp, shape, A, R, prec):
    import torch
    from oracle import dense as od
    m = ci.dense_cp(shape, A, R, 0.9, seed=3)
    dt = torch.float32 if prec == "F32" else torch.float64
    V = np.asarray(ci.random_values(shape, seed=2), dtype=np.float32).reshape(shape).astype(np.float64)
    Q = np.asarray(od.q_values(m, V)).reshape(A, -1)
    f = cp.build_factors(m, device=0)
    Vd = torch.as_tensor(V.reshape(-1)).to("cuda", dt)
    out, pi = torch.empty_like(Vd), torch.zeros(m.nstates, dtype=torch.uint8, device="cuda")
    res = torch.zeros(1, dtype=torch.float64, device="cuda")
    cp.bellman_backup(f, getattr(cp, prec), Vd, out, pi, res)
    u = 2.0 ** (-24 if prec == "F32" else -53)
    tol = (2 * sum(shape) + 8) * u * (np.abs(V).max() + np.abs(m.reward).max())
    got, want = out.double().cpu().numpy(), Q.max(0)
    assert np.abs(got - want).max() <= tol
    chosen = Q[pi.cpu().numpy(), np.arange(m.nstates)]
    assert (want - chosen).max() <= 2 * tol
    assert abs(res.item() - np.abs(got - V.reshape(-1)).max()) <= 1e-6 * res.item()
    f.close()
