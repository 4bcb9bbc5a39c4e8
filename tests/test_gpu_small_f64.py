"""FP64 likelihood and L-BFGS of small problems (several walkers per warp): every lane
grouping gives the same bits, and the values are the oracle's."""
import numpy as np
import pytest

import oracle
import paper_2601_19957_gb300 as sb
from paper_2601_19957_gb300.instances import SolveConfig, make_instance

pytestmark = pytest.mark.gpu

# edges of the groupings (8, 16, 32 lanes a walker) and of their slots; 128 and the K = 8,
# d = 80 case are the largest that take this path (the triangles fill the shared memory)
CASES = [(1, 1), (2, 3), (7, 2), (8, 1), (9, 4), (16, 2), (17, 5), (33, 3), (64, 4), (65, 2), (80, 8), (127, 2),
         (128, 2)]


def _problem(d, K, overlap):
    # overlapping components share responsibility; separated ones are left early
    sep = 0.0 if overlap or d < 8 else 8.0
    box = (-0.3, 0.3) if overlap else (-6, 6)
    inst = make_instance(d, K, 40 + d + K, s_range=(0.2, 0.5), mean_box=box, sep=sep)
    return inst, sb.Problem(inst)


def _oracle(inst, x):
    out = [oracle.loglik(inst, p, want_grad=True) for p in x]
    return np.array([o[0] for o in out]), np.array([o[1] for o in out])


def _points(inst, n, rng):
    k = rng.integers(0, inst.K, n)
    x = inst.mu[k] + rng.standard_normal((n, inst.d)) * 0.3
    x[::5] = rng.uniform(-10, 10, (len(x[::5]), inst.d))
    return np.clip(x, -10, 10)


@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("d,K", CASES)
def test_loglik_same_bits_in_every_grouping(d, K, overlap):
    import torch

    inst, prob = _problem(d, K, overlap)
    x = _points(inst, 3001, np.random.default_rng(d * 10 + K))
    xt = torch.as_tensor(x, device="cuda")
    ell, grad = sb.loglik(prob, xt)
    assert torch.equal(sb.loglik(prob, xt, want_grad=False), ell)
    for i0, n in ((0, 1), (5, 3), (10, 700)):  # 32, 32 and 16 or 8 lanes a point
        e, g = sb.loglik(prob, xt[i0:i0 + n])
        assert torch.equal(e, ell[i0:i0 + n]) and torch.equal(g, grad[i0:i0 + n])
    idx = np.arange(0, 3001, 97)
    rl, rg = _oracle(inst, x[idx])
    np.testing.assert_allclose(ell.cpu().numpy()[idx], rl, rtol=1e-12, atol=1e-12)
    scale = np.abs(rg).max(axis=1, keepdims=True) + 1.0
    assert np.all(np.abs(grad.cpu().numpy()[idx] - rg) <= 1e-12 * scale)


@pytest.mark.parametrize("d,K", [(1, 1), (8, 1), (9, 4), (33, 3), (65, 2)])
def test_refine_same_bits_in_every_grouping(d, K):
    import torch

    inst, prob = _problem(d, K, False)
    starts = torch.as_tensor(_points(inst, 3000, np.random.default_rng(d)), device="cuda")
    cfg = sb.make_config(SolveConfig(n_rays=64, n_steps=64, n_starts=3000, m=6, max_iter=200))
    full = sb.refine(prob, cfg, starts)
    for i0, n in ((3, 1), (20, 40)):
        part = sb.refine(prob, cfg, starts[i0:i0 + n])
        for a, b in ((part.x, full.x), (part.ell, full.ell), (part.status, full.status), (part.iters, full.iters)):
            assert torch.equal(a, b[i0:i0 + n])
    assert int((full.status == sb.RUNNING).sum()) == 0


def test_non_finite_points_stay_local():
    import torch

    inst, prob = _problem(16, 2, False)
    x = _points(inst, 64, np.random.default_rng(0))
    x[7, 3] = np.nan
    x[9, 0] = np.inf
    x[11, 5] = 1e200  # |z|^2 overflows
    ell, grad = sb.loglik(prob, torch.as_tensor(x, device="cuda"))
    ok = np.ones(64, bool)
    ok[[7, 9, 11]] = False
    rl, rg = _oracle(inst, x[ok])
    np.testing.assert_allclose(ell.cpu().numpy()[ok], rl, rtol=1e-12)
    assert np.isfinite(grad.cpu().numpy()[ok]).all()
    assert not np.isfinite(ell.cpu().numpy()[~ok]).any()
