"""The full-grid loss gradient with its arrays at odd addresses (dy on 2 bytes,
resid and V_target on 4): the same bits as with aligned ones, and nothing
written outside them."""
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


@pytest.mark.parametrize("shape", [(4, 4, 4), (10, 9, 7), (16, 20, 68), (17, 66, 65)])
def test_unaligned_equals_aligned(cp, shape):
    import torch
    count, n = 3, int(np.prod(shape))
    cells = int(np.prod([(s + 3) // 4 for s in shape]))
    inst = [ci.gridworld(shape, p=0.8, gamma=0.95, step_reward=-0.01, goal_rewards=[0.6], obstacle_rate=0.15, seed=i)
            for i in range(count)]
    B = cp.batch_build(inst, device=0)
    total = int(B.total_states)
    pred, base = (torch.as_tensor(ci.random_values((count * cells,), seed=s).astype(np.float32)).cuda() for s in (1, 2))
    vt = torch.as_tensor(ci.random_values((total,), seed=3).astype(np.float32)).cuda()
    got = []
    for dy_off, off in ((0, 0), (1, 0), (4, 1), (8, 2)):
        dyb = torch.full((count * cells * 64 + 16,), 7.0, dtype=torch.bfloat16, device="cuda")
        rb = torch.full((count * n + 8,), 7.0, device="cuda")
        vb = torch.zeros(total + 8, device="cuda")
        dy, r, v = dyb[dy_off:dy_off + count * cells * 64], rb[off:off + count * n], vb[off:off + total].copy_(vt)
        cp.ws_fine_loss_grad(B, v, 0, count, pred, base, r, dy, None)
        cp.ws_sync()
        assert (dyb[:dy_off] == 7).all() and (dyb[dy_off + count * cells * 64:] == 7).all()
        assert (rb[:off] == 7).all() and (rb[off + count * n:] == 7).all()
        got.append((dy.view(torch.int16).cpu().numpy().copy(), r.cpu().numpy().copy()))
    for d, r in got[1:]:
        assert np.array_equal(d, got[0][0]) and np.array_equal(r, got[0][1])
    d = got[0][0].reshape(-1, 64)
    assert (d[:, 1:] == 0).all() and (d[:, 0] != 0).any()
    B.close()
