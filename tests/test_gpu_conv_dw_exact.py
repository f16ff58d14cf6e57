"""Weight and bias gradients of whole numbers: every sum stays below 2^24, so
dW and db are exact at any size, and a tile left out, counted twice or taken
from the wrong voxels shows. And of random operands: within 1e-6 of the sum of
|dy x| (8 truncated additions of at most 2^-23 of it in a tile; the additions
after them round to nearest), whatever the number of voxels."""
import numpy as np
import pytest

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


def _sums(x, dy, dims, dil):
    import torch
    n, z, y, xx = dims
    pad = torch.nn.functional.pad(x.double().reshape(*dims, 64), (0, 0) + (dil,) * 6)
    d2 = dy.double().reshape(-1, 64)
    return torch.stack([d2.T @ pad[:, dil * (t // 9):dil * (t // 9) + z, dil * (t // 3 % 3):dil * (t // 3 % 3) + y,
                                   dil * (t % 3):dil * (t % 3) + xx].reshape(-1, 64) for t in range(27)])


@pytest.mark.parametrize("dims,dil", [((1, 1, 1, 1), 1), ((2, 3, 4, 5), 2), ((1, 5, 5, 5), 1), ((1, 5, 17, 33), 1),
                                      ((2, 16, 16, 16), 1), ((7, 16, 16, 16), 1), ((9, 16, 16, 15), 2), ((2, 9, 8, 20), 4),
                                      ((1, 6, 30, 9), 13), ((60, 4, 4, 4), 3), ((32, 16, 16, 16), 1)])
@pytest.mark.parametrize("odd", [0, 1])
def test_weight_gradient(cp, dims, dil, odd):
    import torch
    nv = int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(nv + dil)
    bufs = [torch.empty(nv * 64 + 1, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    x, dy = (b[odd:odd + nv * 64] for b in bufs)
    for whole in (True, False):
        for t in (x, dy):
            t.copy_(torch.randint(-3, 4, (nv * 64,), generator=g, device="cuda") if whole
                    else torch.randn(nv * 64, generator=g, device="cuda"))
        dw, db = torch.zeros(27, 64, 64, device="cuda"), torch.zeros(64, device="cuda")
        cp.conv3d_backward_weight(x, dy, dw, db, dims, dil)
        cp.ws_sync()
        want, db_want = _sums(x, dy, dims, dil), dy.double().reshape(-1, 64).sum(0)
        if whole:
            assert 9 * nv < 1 << 24
            assert torch.equal(dw.double(), want) and torch.equal(db.double(), db_want)
        else:
            mag = _sums(x.abs(), dy.abs(), dims, dil)
            assert ((dw.double() - want).abs() <= 1e-6 * mag).all()
            assert ((db.double() - db_want).abs() <= 1e-6 * dy.double().abs().reshape(-1, 64).sum(0)).all()
