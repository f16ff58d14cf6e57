"""Choices and certificates of the FP64 backup that depend on how values are
widened and compared: denormal floats, zeros of both signs, infinities, NaN.

Weights (p and the slip share) are powers of two or small multiples of them
and values short, so every expectation is exact and the documented rule - the
larger neighbour of each dimension, the first on ties and where a comparison
with a NaN is false; then the first dimension with the largest expectation -
gives one action per state. Residuals skip NaN."""
import numpy as np
import pytest

import cpmdp_inputs as ci

pytestmark = pytest.mark.gpu

P = {2: 0.75, 3: 0.75, 4: 0.625, 5: 0.75}     # (1 - p) / (2 (D - 1)): 1/8, 1/16, 1/16, 1/32


@pytest.fixture(scope="module")
def cp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build_library()
    import paper_2103_00331_gb300 as cp
    return cp


def _rule(gw, V):
    """(R + gamma E, action) of every state as if free, FP64."""
    shape, D = gw.shape, len(gw.shape)
    V = V.reshape(shape)
    obst = np.asarray(gw.cell).reshape(shape) == ci.OBSTACLE
    nb = []
    for d in range(D):
        for sg in (-1, 1):
            bad = np.roll(obst, -sg, d)
            edge = [slice(None)] * D
            edge[d] = -1 if sg > 0 else 0
            bad[tuple(edge)] = True
            nb.append(np.where(bad, V, np.roll(V, -sg, d)))
    wp = (1 - gw.p) / (2 * (D - 1))
    with np.errstate(all="ignore"):
        pair = [nb[2 * d] + nb[2 * d + 1] for d in range(D)]
        best = arg = None
        for d in range(D):
            up = nb[2 * d + 1] > nb[2 * d]
            e = gw.p * np.where(up, nb[2 * d + 1], nb[2 * d]) + wp * sum(pair[j] for j in range(D) if j != d)
            a = 2 * d + up
            if best is None:
                best, arg = e, a
            else:
                take = e > best
                best, arg = np.where(take, e, best), np.where(take, a, arg)
        return (np.asarray(gw.reward).reshape(shape) + gw.gamma * best).reshape(-1), arg.reshape(-1)


def _world(shape, seed=3):
    return ci.gridworld(shape, p=P[len(shape)], gamma=0.5, step_reward=-0.25, goal_rewards=[1.0], obstacle_rate=0.1,
                        seed=seed)


def _residual(gw, want, V):
    cell = np.asarray(gw.cell).reshape(-1)
    want = np.where(cell == ci.TERMINAL, np.asarray(gw.reward).reshape(-1), want)
    with np.errstate(all="ignore"):
        dv = np.abs(want - V)[cell != ci.OBSTACLE]
    return 0.0 if np.isnan(dv).all() else np.nanmax(dv)


@pytest.mark.parametrize("shape", [(10, 10), (9, 13), (64, 66), (5, 6, 7), (12, 8, 16), (3, 4, 5, 6), (3, 2, 3, 2, 3)])
@pytest.mark.parametrize("kind", ["zeros", "ties", "inf", "nan"])
def test_fp64_actions(cp, shape, kind):
    import torch
    gw = _world(shape)
    n = gw.nstates
    V = np.floor(ci.random_values(shape, seed=7, lo=-2, hi=2).reshape(-1))
    pick = ci.integers(5, 1, n, 0, 4)
    if kind == "zeros":
        V = np.where(pick < 2, 0.0, np.where(pick == 2, -0.0, V))
    elif kind == "inf":
        V = np.where(pick == 0, np.inf, np.where(ci.integers(6, 1, n, 0, 30) == 0, -np.inf, V))
    elif kind == "nan":
        V = np.where(ci.integers(6, 1, n, 0, 12) == 0, np.where(pick < 2, np.nan, -np.nan), V)
    f = cp.build_factors(gw, device=0)
    Vd = torch.as_tensor(V, device="cuda")
    out = torch.empty_like(Vd)
    pi = torch.full((n,), 99, dtype=torch.uint8, device="cuda")
    cp.bellman_backup(f, cp.F64, Vd, out, pi, None)
    want, arg = _rule(gw, V)
    free = np.asarray(gw.cell).reshape(-1) == ci.FREE
    assert np.array_equal(pi.cpu().numpy()[free], arg[free])
    assert np.array_equal(out.cpu().numpy()[free], want[free], equal_nan=True)
    f.close()


# the last: past the size from which 3-D sweeps march over planes
@pytest.mark.parametrize("shape", [(10, 12), (17, 19), (6, 7, 8), (16, 16, 16), (31, 29, 33), (4, 5, 6, 4), (200, 208, 212)])
@pytest.mark.parametrize("kind", ["denormal", "inf", "nan"])
def test_certificate(cp, shape, kind):
    """One FP32 sweep and its FP64 certificate: residual and actions of the
    returned floats. Denormal: rewards, and so values and residual, of a few
    times 1e-45 (whole multiples of the smallest float)."""
    import torch
    gw = _world(shape)
    n = gw.nstates
    r = np.asarray(gw.reward).reshape(-1)
    V = np.zeros(n, dtype=np.float32)
    if kind == "denormal":
        tiny = 2.0 ** -149
        r[:] = np.where(np.asarray(gw.cell).reshape(-1) == ci.OBSTACLE, 0.0, tiny * 16 * ci.integers(9, 1, n, -40, 41))
    else:
        V = np.round(ci.random_values(shape, seed=7, lo=-2, hi=2).reshape(-1)).astype(np.float32)
        V[ci.integers(6, 1, n, 0, 40) == 0] = np.inf if kind == "inf" else np.nan
    f = cp.build_factors(gw, device=0)
    Vd = torch.as_tensor(V).cuda()
    pi = torch.full((n,), 99, dtype=torch.uint8, device="cuda")
    info = cp.value_iteration(f, cp.F32, Vd, pi, opts=cp.default_opts(max_iter=1), raise_on_noconv=False)
    Vh = Vd.double().cpu().numpy()
    want, arg = _rule(gw, Vh)
    far = _residual(gw, want, Vh)
    free = np.asarray(gw.cell).reshape(-1) == ci.FREE
    if kind == "denormal":
        assert 0.0 < far < 1e-40 and (Vh != 0).any()
    assert np.array_equal(pi.cpu().numpy()[free], arg[free])
    assert info["certified_residual"] == far
    f.close()


@pytest.mark.parametrize("kind", ["denormal", "inf", "nan"])
def test_batch_certificate(cp, kind):
    import torch
    shapes = [(10, 12), (9, 13), (6, 7, 8), (16, 16, 16)]
    inst = [_world(s, seed=3 + i) for i, s in enumerate(shapes)]
    tiny = 2.0 ** -149
    for i, gw in enumerate(inst):
        if kind == "denormal":
            np.asarray(gw.reward).reshape(-1)[:] = np.where(np.asarray(gw.cell).reshape(-1) == ci.OBSTACLE, 0.0,
                                                            tiny * 16 * ci.integers(9, i, gw.nstates, -40, 41))
    B = cp.batch_build(inst, device=0)
    V = torch.zeros(int(B.total_states), dtype=torch.float32, device="cuda")
    host = []
    for i, gw in enumerate(inst):
        n, at = gw.nstates, int(B.offsets[i])
        v = np.round(ci.random_values(gw.shape, seed=7, lo=-2, hi=2).reshape(-1))
        if kind == "denormal":
            v = tiny * 16 * ci.integers(11, i, n, -40, 41)
        else:
            v[ci.integers(6, i, n, 0, 40) == 0] = np.inf if kind == "inf" else np.nan
        host.append(v)
        V[at:at + n] = torch.as_tensor(v.astype(np.float32))
    pi = torch.full((int(B.total_states),), 99, dtype=torch.uint8, device="cuda")
    res = cp.batch_certify(B, V, pi)
    for i, gw in enumerate(inst):
        want, arg = _rule(gw, host[i])
        free = np.asarray(gw.cell).reshape(-1) == ci.FREE
        at = int(B.offsets[i])
        assert np.array_equal(pi.cpu().numpy()[at:at + gw.nstates][free], arg[free])
        assert res[i] == _residual(gw, want, host[i])
    B.close()
