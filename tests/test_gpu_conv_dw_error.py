"""Error of the warm-start convolution's weight gradient against FP64: the
tensor-core kernel (16-byte aligned operands) is no further off than the FP32
pipe (the same operands at an odd address), in the root mean square over all
outputs, from grids of a few tiles to a minibatch. x is positive, as after a
ReLU, and dy has a mean, so that truncated sums drift one way."""
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


def _dw64(x, dy, dims):
    import torch
    n, z, y, xx = dims
    pad = torch.nn.functional.pad(x.double().reshape(*dims, 64), (0, 0) + (1,) * 6)
    d2 = dy.double().reshape(-1, 64)
    return torch.stack([d2.T @ pad[:, t // 9:t // 9 + z, t // 3 % 3:t // 3 % 3 + y, t % 3:t % 3 + xx].reshape(-1, 64)
                        for t in range(27)])


@pytest.mark.parametrize("dims", [(1, 4, 4, 4), (4, 5, 5, 5), (4, 8, 8, 8), (1, 16, 16, 16), (2, 16, 16, 16),
                                  (4, 16, 16, 16), (8, 16, 16, 16)])
def test_no_further_off_than_fp32(cp, dims):
    import torch
    nv = int(np.prod(dims))
    square = [0.0, 0.0]
    for seed in range(4):
        g = torch.Generator(device="cuda").manual_seed(100 * seed + nv)
        xr = torch.randn(nv * 64, generator=g, device="cuda").relu().to(torch.bfloat16)
        dr = (torch.randn(nv * 64, generator=g, device="cuda") * 1e-3 + 5e-4).to(torch.bfloat16)
        want = _dw64(xr, dr, dims)
        for odd in (0, 1):
            bufs = [torch.empty(nv * 64 + 1, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
            x, dy = (b[odd:odd + nv * 64].copy_(v) for b, v in zip(bufs, (xr, dr)))
            dw = torch.zeros(27, 64, 64, device="cuda")
            cp.conv3d_backward_weight(x, dy, dw, None, dims, 1)
            cp.ws_sync()
            square[odd] += (dw.double() - want).square().mean().item()
    assert square[0] <= square[1] * 1.01      # reductions land in any order: a percent of either
