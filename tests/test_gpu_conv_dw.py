"""Weight and bias gradients of the warm-start convolution: the tensor-core
kernel (tile shapes with and without the shared y rows, tiles cut short, one
and two ring stages, dilations past the grid) and the FP32 form that unaligned
operands take, against the same sums in FP64.

Tolerance: products of bf16 values are exact in FP32, so each output is off by
at most the rounding of its additions: (number of voxels + 64) 2^-23 times the
sum of |dy x| over its voxels (2^-23 covers truncating adders).
"""
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


def _sums(x, dy, dil):
    """FP64 dW and the sums of absolute values, [27, co, ci]."""
    import torch
    n, z, y, xx, c = x.shape
    pad = torch.nn.functional.pad(x, (0, 0) + (dil,) * 6)
    d2 = dy.reshape(-1, c)
    out, mag = [], []
    for t in range(27):
        oz, oy, ox = dil * (t // 9), dil * (t // 3 % 3), dil * (t % 3)
        part = pad[:, oz:oz + z, oy:oy + y, ox:ox + xx].reshape(-1, c)
        out.append(d2.T @ part)
        mag.append(d2.abs().T @ part.abs())
    return torch.stack(out), torch.stack(mag)


@pytest.mark.parametrize("dims,dil", [((1, 1, 1, 1), 1), ((2, 3, 4, 5), 2), ((1, 5, 17, 33), 1), ((7, 16, 16, 16), 1),
                                      ((3, 16, 16, 16), 2), ((2, 9, 8, 20), 4), ((1, 6, 30, 9), 13), ((60, 4, 4, 4), 3)])
@pytest.mark.parametrize("odd", [0, 1])
def test_weight_gradient(cp, dims, dil, odd):
    import torch
    nv = int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(nv + dil)
    bufs = [torch.randn(nv * 64 + 1, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
    x, dy = (b[odd:odd + nv * 64] for b in bufs)       # odd: 2-byte aligned only
    dw = torch.full((27, 64, 64), 0.5, device="cuda")   # the call adds
    db = torch.full((64,), -0.25, device="cuda")
    cp.conv3d_backward_weight(x, dy, dw, db, dims, dil)
    cp.ws_sync()
    want, mag = _sums(x.double().reshape(*dims, 64), dy.double().reshape(*dims, 64), dil)
    tol = (nv + 64) * 2.0 ** -23
    assert ((dw.double() - 0.5 - want).abs() <= tol * (mag + 0.5)).all()
    d2 = dy.double().reshape(-1, 64)
    assert ((db.double() + 0.25 - d2.sum(0)).abs() <= tol * (d2.abs().sum(0) + 0.25)).all()
