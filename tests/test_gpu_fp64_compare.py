"""FP64 backups whose comparisons run on the integer pipe: zeros of both signs,
ties, denormals, infinities and NaN among the values give what floating-point
comparisons give, and FP32 values widen exactly (the FP64 certificate).

The reference applies the documented rule per state in numpy: for each
dimension the larger neighbour (the first on ties and where the comparison
with a NaN is false), E = p m + slip sum of the other pairs, the first largest
E. Finite values agree to 4 ulp of (max|R| + max|V|) (one fused product may
round differently); where the rule gives NaN or an infinity the backup does."""
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


def _rule(gw, V):
    shape, D = gw.shape, len(gw.shape)
    V = V.reshape(shape)
    obst = np.asarray(gw.cell).reshape(shape) == ci.OBSTACLE
    nb = []
    for d in range(D):
        for sg in (-1, 1):
            x = np.roll(V, -sg, d)
            bad = np.roll(obst, -sg, d)
            edge = [slice(None)] * D
            edge[d] = -1 if sg > 0 else 0
            bad[tuple(edge)] = True
            nb.append(np.where(bad, V, x))
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
        out = np.asarray(gw.reward).reshape(shape) + gw.gamma * best
    return out.reshape(-1), arg.reshape(-1)


@pytest.mark.parametrize("shape", [(10, 10), (9, 13), (64, 66), (5, 6, 7), (12, 8, 16), (3, 4, 5, 6), (3, 2, 3, 2, 3)])
@pytest.mark.parametrize("kind", ["zeros", "ties", "denormal", "inf", "nan"])
def test_fp64_backup_special_values(cp, shape, kind):
    import torch
    gw = ci.gridworld(shape, p=0.75, gamma=0.5, step_reward=-0.25, goal_rewards=[1.0], obstacle_rate=0.1, seed=3)
    n = gw.nstates
    V = ci.random_values(shape, seed=7, lo=-2, hi=2).reshape(-1)
    pick = ci.integers(5, 1, n, 0, 4)
    if kind == "zeros":
        V = np.where(pick < 2, 0.0, np.where(pick == 2, -0.0, V))
    elif kind == "ties":
        V = np.round(V)
    elif kind == "denormal":
        V = np.where(pick == 0, 5e-324, np.where(pick == 1, -1e-310, np.where(pick == 2, 0.0, V * 1e-308)))
    elif kind == "inf":
        V = np.where(pick == 0, np.inf, np.where(ci.integers(6, 1, n, 0, 30) == 0, -np.inf, V))
    else:
        V = np.where(ci.integers(6, 1, n, 0, 12) == 0, np.nan, V)
    f = cp.build_factors(gw, device=0)
    Vd = torch.as_tensor(V, device="cuda")
    out = torch.empty_like(Vd)
    out2 = torch.empty_like(Vd)
    pi = torch.zeros(n, dtype=torch.uint8, device="cuda")
    res = torch.zeros(1, dtype=torch.float64, device="cuda")
    cp.bellman_backup(f, cp.F64, Vd, out, pi, res)
    cp.bellman_backup(f, cp.F64, Vd, out2, None, None)
    torch.cuda.synchronize()
    want, arg = _rule(gw, V)
    free = np.asarray(gw.cell).reshape(-1) == ci.FREE
    got, got2, pol = out.cpu().numpy(), out2.cpu().numpy(), pi.cpu().numpy()
    fin = np.isfinite(want) & free
    tol = 4 * 2.0 ** -52 * (1.0 + np.abs(V[np.isfinite(V)]).max())
    for g in (got, got2):
        assert np.abs(g[fin] - want[fin]).max(initial=0.0) <= tol
        assert np.array_equal(np.isnan(g[free]), np.isnan(want[free]))
        assert np.array_equal(g[free & np.isinf(want)], want[free & np.isinf(want)])
    if kind in ("ties", "zeros"):
        # exact small integers times 0.75 and a power of two of it: no rounding, so ties are ties
        if kind == "ties" and len(shape) == 2:
            assert np.array_equal(pol[free], arg[free])
    live = np.asarray(gw.cell).reshape(-1) != ci.OBSTACLE
    with np.errstate(all="ignore"):
        dv = np.abs(got - V)[live]
    assert res.item() == (np.nanmax(dv) if np.any(~np.isnan(dv)) else 0.0)
    f.close()


@pytest.mark.parametrize("shape", [(10, 12), (6, 7, 8), (16, 16, 16), (4, 5, 6, 4)])
def test_certificate_widens_exactly(cp, shape):
    """One sweep of FP32 value iteration, then its FP64 certificate: the
    residual of the returned floats (denormals and zeros among them)."""
    import torch
    gw = ci.gridworld(shape, p=0.75, gamma=0.5, step_reward=-0.25, goal_rewards=[1.0], obstacle_rate=0.1, seed=3)
    r = np.asarray(gw.reward).reshape(-1)
    r[::5] = 0.0
    r[1::7] = -1e-41
    r[np.asarray(gw.cell).reshape(-1) == ci.OBSTACLE] = 0.0
    f = cp.build_factors(gw, device=0)
    V = torch.zeros(gw.nstates, dtype=torch.float32, device="cuda")
    pi = torch.zeros(gw.nstates, dtype=torch.uint8, device="cuda")
    a = cp.value_iteration(f, cp.F32, V, pi, opts=cp.default_opts(max_iter=1), raise_on_noconv=False)
    Vh = V.double().cpu().numpy()
    want, _ = _rule(gw, Vh)
    cell = np.asarray(gw.cell).reshape(-1)
    want = np.where(cell == ci.TERMINAL, r, want)
    dv = np.abs(want - Vh)[cell != ci.OBSTACLE].max()
    assert abs(a["certified_residual"] - dv) <= 4 * 2.0 ** -52 * 2.0
    f.close()
