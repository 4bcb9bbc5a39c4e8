"""Indefinite Hessians beside good ones in one blocked factorisation: a candidate whose pivot
turns negative in some block must leave the others' results as they are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2601_19957_gb300 as sb
from paper_2601_19957_gb300.instances import SolveConfig, make_instance

pytestmark = pytest.mark.gpu


def _pairs(d, axes, seed):
    """Components in pairs 6 apart along the given axes: half way between the two of a pair
    the factorisation fails at that coordinate (curvature 1 - 9), the blocks before it pass."""
    K = 2 * len(axes)
    inst = make_instance(d, K, seed, s_range=(1.0, 1.0), sep=0.0)
    rng = np.random.default_rng(seed)
    low = np.eye(d) + np.tril(rng.standard_normal((d, d)), -1) * (0.1 / d)
    mid = np.zeros((len(axes), d))
    for p, j in enumerate(axes):
        mid[p, 0], mid[p, 1] = (-7.0, 0.0, 7.0)[p % 3], (-7.0, 0.0, 7.0)[p // 3 % 3]
        for q, s in enumerate((-3.0, 3.0)):
            inst.mu[2 * p + q] = mid[p]
            inst.mu[2 * p + q, j] += s
            inst.L[2 * p + q] = low
    inst.log_w[:] = np.log(1.0 / K)
    return inst, mid


@pytest.mark.parametrize("d,axes", [
    (40, (35,)),                                  # the last, short block
    (70, (33, 66)),
    (96, (40, 70, 95)),                           # the first to the last block after the diagonal's first
    (160, (20, 50, 90, 130, 159)),                # one fails in the first block
    (512, (40, 100, 200, 300, 400, 450, 480, 511)),
])
def test_saddles_beside_modes_leave_the_modes_as_they_are(d, axes):
    inst, mid = _pairs(d, axes, 3 + d)
    prob = sb.Problem(inst)
    rng = np.random.default_rng(d)
    near = inst.mu + 0.01 * rng.standard_normal(inst.mu.shape)
    c = SolveConfig(n_rays=1, n_steps=1, n_starts=1, cand_cap=64, newton_steps=6)
    cfg = sb.make_config(c)

    def run(x):
        t = torch.as_tensor(np.ascontiguousarray(x), device="cuda")
        return sb.laplace(prob, cfg, t, sb.loglik(prob, t, want_grad=False))

    good = run(near)
    ref = oracle.laplace(inst, c, near, np.array([oracle.loglik(inst, x) for x in near]))
    assert good.n_modes == ref.n_modes == inst.K
    assert np.allclose(good.logZk.cpu().numpy(), ref.logZk, rtol=0, atol=1e-10)
    assert run(mid).n_modes == 0
    for _ in range(5):
        both = run(np.concatenate([mid, near]))
        assert both.n_modes == good.n_modes
        assert torch.equal(both.modes, good.modes) and torch.equal(both.logZk, good.logZk)
        assert both.logZ == good.logZ
