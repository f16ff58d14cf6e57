"""Dense sweeps and policy iteration through every form of the fused chains:
both register tiles of the last run of modes, FP32 and FP64, and models whose
intermediates exceed 1 GiB, so that the running maximum, its action and the
kept action's Q pass from one group of actions to the next.

The models move most of the mass along a shift of each mode that depends on
the action (uniform noise for the rest, the first rank term weighted most), so
that actions differ by far more than rounding. Reference: the same in FP64,
plain torch. One sweep: FP64 1e-12 (max|R| + max|V|), FP32
(sum_d (N_d + 2) + R + 4) 2^-24 of it =: eps. Policy iteration stops with
|T V - V| <= eval_tol + margin + 3 eps (evaluated policy within eval_tol, no
action better by more than the margin 1e-6 (1e-12) (1 + |Q|), rounding of
three sweeps), so |V - V*| is below that over 1 - gamma.
"""
from types import SimpleNamespace

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


def _model(shape, A, R, gamma):
    rng = np.random.default_rng([A, R, *shape])
    parts = []
    for a in range(A):
        for r in range(R):
            for d, n in enumerate(shape):
                m = rng.random((n, n))
                m *= 0.1 / m.sum(axis=1, keepdims=True)
                i = np.arange(n)
                m[i, (i + (a >> d) * (1 + d) + 3 * r) % n] += 0.9
                parts.append(m.ravel())
    lam = 0.6 ** np.arange(R)
    packed = np.concatenate(parts)
    return SimpleNamespace(shape=shape, nactions=A, rank=R, lam=np.tile(lam / lam.sum(), (A, 1)), gamma=gamma,
                           reward=rng.standard_normal(int(np.prod(shape))), packed=packed,
                           packed_factors=lambda: packed)


class Reference:
    def __init__(self, m):
        import torch
        self.m, self.torch = m, torch
        self.R = torch.as_tensor(m.reward).cuda()
        self.U = torch.as_tensor(m.packed).cuda().view(m.nactions, m.rank, -1)
        self.lam = torch.as_tensor(m.lam).cuda()

    def q(self, V):
        """Q[a, s], one action at a time."""
        m = self.m
        for a in range(m.nactions):
            x, off = V.view(1, *m.shape).expand(m.rank, *m.shape), 0
            for d, n in enumerate(m.shape):
                u = self.U[a, :, off:off + n * n].reshape(m.rank, 1, n, n)
                off += n * n
                x = u @ x.reshape(m.rank, int(np.prod(m.shape[:d])), n, -1)
            yield self.R + m.gamma * (self.lam[a] @ x.reshape(m.rank, -1))

    def backup(self, V):
        """Largest Q, its first action, and the distance to the second largest."""
        torch = self.torch
        best = arg = second = None
        for a, q in enumerate(self.q(V)):
            if best is None:
                best, arg, second = q, torch.zeros_like(q, dtype=torch.uint8), torch.full_like(q, -np.inf)
                continue
            take = q > best
            second = torch.where(take, best, torch.maximum(second, q))
            best = torch.where(take, q, best)
            arg[take] = a
        return best, arg, best - second

    def optimum(self):
        V = self.torch.zeros_like(self.R)
        for _ in range(400):
            W = self.backup(V)[0]
            far = (W - V).abs().max().item()
            V = W
            if far < 1e-12:
                return V
        raise AssertionError("no convergence")


MODELS = [((5,), 2, 2), ((33, 47), 3, 4), ((20, 21, 9), 4, 3), ((30, 31, 29), 5, 1), ((30, 30, 30, 30), 4, 4),
          ((2, 3, 2, 3, 2), 3, 1),
          ((41, 41, 41), 64, 64),       # FP32 two groups of actions (narrow tile), FP64 three
          ((30, 30, 30, 30), 8, 64)]    # FP32 two groups (wide tile), FP64 four


@pytest.mark.parametrize("shape,A,R", MODELS)
def test_sweep_and_policy_iteration(cp, shape, A, R):
    import torch
    m = _model(shape, A, R, 0.5)
    ref = Reference(m)
    n = m.reward.size
    Vs = ref.optimum()
    _, pis, gap = ref.backup(Vs)
    f = cp.build_factors(m, device=0)
    for prec, dt, eval_tol, unit in ((cp.F32, torch.float32, 1e-6, 1e-6), (cp.F64, torch.float64, 1e-10, 1e-12)):
        g = torch.Generator(device="cuda").manual_seed(n)
        V = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 4 - 2).to(dt)
        scale = np.abs(m.reward).max() + max(2.0, Vs.abs().max().item())
        eps = 1e-12 * scale if prec == cp.F64 else (sum(s + 2 for s in shape) + R + 4) * 2.0 ** -24 * scale
        # one sweep
        out = torch.full((n,), float("nan"), dtype=dt, device="cuda")
        pi = torch.full((n,), 99, dtype=torch.uint8, device="cuda")
        res = torch.zeros(1, dtype=torch.float64, device="cuda")
        cp.bellman_backup(f, prec, V, out, pi, res)
        want, arg, near = ref.backup(V.double())
        assert (out.double() - want).abs().max().item() <= eps
        sure = near > 2 * eps
        assert sure.double().mean().item() > 0.5
        assert torch.equal(pi[sure], arg[sure])
        assert res.item() == (out.double() - V.double()).abs().max().item()
        # policy iteration: greedy, evaluation and improvement sweeps
        margin = unit * (1 + scale)
        bound = (eval_tol + margin + 3 * eps) / (1 - m.gamma)
        V.zero_()
        r = cp.policy_iteration(f, prec, V, pi)
        assert r["status"] == cp.OK and r["rounds"] >= 1
        assert (V.double() - Vs).abs().max().item() <= bound
        sure = gap > 2 * m.gamma * bound + margin + 2 * eps
        assert sure.double().mean().item() > 0.5
        assert torch.equal(pi[sure], pis[sure])
    f.close()
