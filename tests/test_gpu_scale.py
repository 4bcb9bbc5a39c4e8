"""Problems scaled by powers of two: FP32 routes of FP64 decisions hold at every scale."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2601_19957_gb300 as sb
from paper_2601_19957_gb300.instances import SolveConfig, make_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exp", [-140, -60, 100])
def test_duplicates_are_merged_alike_at_every_scale(exp):
    """A problem scaled by a power of two has the scaled modes, in the same number."""
    d, K = 6, 3
    inst = make_instance(d, K, 21, s_range=(0.2, 0.4), mean_box=(-6, 6), sep=8.0)
    rng = np.random.default_rng(4)
    # walkers around each mean within and beyond the merging distance (1e-3 of the box: 0.02)
    x = np.repeat(inst.mu, 40, axis=0) + rng.uniform(-0.03, 0.03, (40 * K, d))
    c = sb.make_config(SolveConfig(n_rays=1, n_steps=1, n_starts=1, cand_cap=200, newton_steps=0, eps_grad=1e9))
    ell = np.array([oracle.loglik(inst, p) for p in x])
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    one = sb.laplace(sb.Problem(inst), c, t(x), t(ell))
    assert one.n_modes > K
    s = 2.0 ** exp
    inst.mu, inst.lo, inst.hi, inst.L = inst.mu * s, inst.lo * s, inst.hi * s, inst.L / s
    c.eps_grad = 1e9 / min(s, 1.0)
    two = sb.laplace(sb.Problem(inst), c, t(x * s), t(ell))
    assert two.n_modes == one.n_modes
    assert torch.equal(two.modes, one.modes * s)


@pytest.mark.parametrize("j", [1, 2, 3, 32, 33, 63])
def test_probe_of_coordinates_before_an_overflowing_one(j):
    """A component whose z overflows at coordinate j (its term is -inf, its weight 0) leaves
    the sensitivities of the coordinates before j as without it."""
    d = 64
    inst = make_instance(d, 2, 8, s_range=(0.3, 1.0), mean_box=(-2, 2), sep=0.0)
    inst.L[1] = np.eye(d)
    inst.L[1, j, j] = 1e160
    inst.mu[1, j] = -1e160
    got = sb.precheck(sb.Problem(inst)).s.cpu().numpy()
    inst.K, inst.log_w, inst.mu, inst.L = 1, inst.log_w[:1], inst.mu[:1], inst.L[:1]
    want = sb.precheck(sb.Problem(inst)).s.cpu().numpy()
    assert np.isfinite(want).all()
    np.testing.assert_allclose(got[:j], want[:j], rtol=1e-10)
