"""Weight gradient of operands that are not finite, most of it in grids that are a
multiple of no tile: an infinity or a NaN of x reaches the taps that pair its
voxel with one of dy in the grid, and no others (the FP32 form, for odd
addresses, likewise). Against the same sums in FP64; the finite ones within
1e-6 of the sum of |dy x|, as for finite operands."""
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
    pad = torch.nn.functional.pad(x.reshape(*dims, 64), (0, 0) + (dil,) * 6)
    out = torch.zeros(27, 64, 64, dtype=torch.float64)
    for t in range(27):
        part = pad[:, dil * (t // 9):dil * (t // 9) + z, dil * (t // 3 % 3):dil * (t // 3 % 3) + y,
                   dil * (t % 3):dil * (t % 3) + xx].reshape(-1, 64)
        for c in range(64):                            # term by term: 0 times infinity is a NaN
            out[t, c] = (dy.reshape(-1, 64)[:, c, None] * part).sum(0)
    return out


@pytest.mark.parametrize("dims,dil", [((2, 5, 5, 5), 1), ((1, 5, 17, 33), 1), ((3, 9, 8, 20), 2), ((8, 15, 15, 15), 1),
                                      ((1, 16, 16, 16), 1)])
@pytest.mark.parametrize("odd", [0, 1])
def test_not_finite(cp, dims, dil, odd):
    import torch
    n, z, y, xx = dims
    nv = int(np.prod(dims))
    g = torch.Generator().manual_seed(nv + dil)
    xh, dh = (torch.randn(nv, 64, generator=g).to(torch.bfloat16) for _ in range(2))
    faces = [(z - 1, y // 2, xx // 2), (z // 2, y - 1, xx // 2), (z // 2, y // 2, xx - 1), (z - 1, y - 1, xx - 1), (0, 0, 0)]
    for c, (at, v) in enumerate((at, v) for at in faces for v in (float("inf"), float("-inf"), float("nan"))):
        xh[((n - 1) * z + at[0]) * y * xx + at[1] * xx + at[2], 4 * c] = v
    dh[(z * y - 1) * xx + xx // 2, 7] = float("inf")
    bufs = [torch.empty(nv * 64 + 1, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    x, dy = (b[odd:odd + nv * 64].copy_(v.reshape(-1)) for b, v in zip(bufs, (xh, dh)))
    dw = torch.zeros(27, 64, 64, device="cuda")
    cp.conv3d_backward_weight(x, dy, dw, None, dims, dil)
    cp.ws_sync()
    got, want = dw.double().cpu(), _sums(xh.double(), dh.double(), dims, dil)
    assert torch.equal(got.isnan(), want.isnan())
    assert torch.equal(got.isposinf(), want.isposinf()) and torch.equal(got.isneginf(), want.isneginf())
    ok = want.isfinite()
    mag = _sums(xh.double().abs(), dh.double().abs(), dims, dil)
    assert ((got - want).abs()[ok] <= 1e-6 * mag[ok]).all()
