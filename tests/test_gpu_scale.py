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
