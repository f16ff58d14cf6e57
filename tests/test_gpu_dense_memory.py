"""Device memory of dense models on the GPU: the build leaves the fused sweeps'
intermediates to the first sweep, which may be one under a stream capture."""
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


def test_build_takes_no_intermediates(cp):
    """30^4, 4 actions, rank 16: 64 intermediates of 3.24 MB in FP32 (198 MiB).
    The build stays below 64 MiB, the first FP32 sweep takes them, the second nothing."""
    import torch
    dc = ci.dense_cp((30, 30, 30, 30), 4, 16, 0.9, seed=1)
    n = dc.nstates
    cp.build_factors(ci.dense_cp((6, 5), 2, 1, 0.9, seed=1), device=0).close()   # modules loaded
    V = torch.as_tensor(ci.random_values(dc.shape, seed=2).reshape(-1).astype(np.float32)).cuda()
    out = torch.empty_like(V)
    free = []
    torch.cuda.synchronize()
    free.append(torch.cuda.mem_get_info()[0])
    f = cp.build_factors(dc, device=0)
    free.append(torch.cuda.mem_get_info()[0])
    for _ in range(2):
        cp.bellman_backup(f, cp.F32, V, out)
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    f.close()
    assert free[0] - free[1] < 64 << 20
    assert free[1] - free[2] >= 64 * n * 4
    assert free[3] == free[2]


@pytest.mark.parametrize("prec", [0, 1])
def test_first_sweep_under_capture(cp, prec):
    import torch
    dc = ci.dense_cp((20, 21, 9), 4, 3, 0.95, seed=5)
    n = dc.nstates
    dt = torch.float64 if prec == cp.F64 else torch.float32
    V = torch.as_tensor(ci.random_values(dc.shape, seed=1).reshape(-1)).to("cuda", dt)
    got = []
    for captured in (True, False):
        f = cp.build_factors(dc, device=0)
        out = torch.zeros(n, dtype=dt, device="cuda")
        pi = torch.full((n,), 99, dtype=torch.uint8, device="cuda")
        res = torch.zeros(1, dtype=torch.float64, device="cuda")
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                cp.bellman_backup(f, prec, V, out, pi, res, stream=torch.cuda.current_stream())
            g.replay()
        else:
            cp.bellman_backup(f, prec, V, out, pi, res)
        torch.cuda.synchronize()
        got.append((out.cpu().numpy(), pi.cpu().numpy(), res.item()))
        f.close()
    assert got[0][2] == got[1][2] and all(np.array_equal(a, b) for a, b in zip(got[0][:2], got[1][:2]))
