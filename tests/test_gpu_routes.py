"""Routes chosen by size: each must give what the general route gives (the same bits where
the sums keep their order, else to rounding)."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2601_19957_gb300 as sb
from paper_2601_19957_gb300.instances import SolveConfig, make_instance

pytestmark = pytest.mark.gpu


def _mixture(d, K, overlap, seed=0):
    if overlap:
        return make_instance(d, K, 70 + d + K + seed, s_range=(0.2, 0.5), mean_box=(-0.2, 0.2), sep=0.0)
    return make_instance(d, K, 70 + d + K + seed, s_range=(0.1, 0.5), mean_box=(-6, 6), sep=8.0)


def _points(inst, n, seed):
    """Near the components, far from all of them, and exactly at the means."""
    rng = np.random.default_rng(seed)
    x = inst.mu[rng.integers(0, inst.K, n)] + rng.standard_normal((n, inst.d)) * rng.choice([0.01, 0.3, 2.0], (n, 1))
    x[::7] = rng.uniform(-10, 10, x[::7].shape)
    x[:inst.K] = inst.mu[: len(x[:inst.K])]
    return torch.as_tensor(np.clip(x, -10, 10), device="cuda")


def _loglik(prob, x, prec, ws_bytes):
    """sb_loglik on a workspace of exactly ws_bytes."""
    n = x.shape[0]
    ell = torch.empty(n, dtype=torch.float64, device="cuda")
    grad = torch.empty_like(x)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    code = sb.lib().sb_loglik(C.byref(prob.s), C.c_int32(prec), sb._ptr(x), C.c_int32(n), sb._ptr(ell), sb._ptr(grad),
                              C.c_void_p(ws.data_ptr()), C.c_size_t(ws_bytes), sb._stream())
    return code, ell, grad


@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("d,K,n", [(129, 2, 256), (200, 5, 333), (256, 8, 1000), (300, 3, 257), (1024, 2, 300)])
def test_fp64_grouped_rows_same_bits_as_every_row(d, K, n, overlap):
    inst = _mixture(d, K, overlap)
    prob = sb.Problem(inst)
    x = _points(inst, n, d)
    full = int(sb.lib().sb_loglik_workspace_bytes(C.byref(prob.s), 0, n))
    lists = 4 * (4 * n + 3 * K * n + 3 * K + 4)  # the row lists come last in the workspace
    code, ell, grad = _loglik(prob, x, 0, full)
    assert code == sb.SB_OK
    code, e0, g0 = _loglik(prob, x, 0, (full - lists) // 256 * 256)  # no room for the lists: accepted
    assert code == sb.SB_OK
    assert torch.equal(ell, e0) and torch.equal(grad, g0)
    assert torch.equal(sb.loglik(prob, x, want_grad=False), ell)
    few = 40  # the matrix-vector kernels: another order
    e1, g1 = sb.loglik(prob, x[:few].contiguous())
    np.testing.assert_allclose(e1.cpu().numpy(), ell[:few].cpu().numpy(), rtol=1e-13, atol=1e-11)
    scale = g1.abs().amax(1, keepdim=True) + 1.0
    assert bool(((g1 - grad[:few]).abs() <= 1e-12 * scale).all())


@pytest.mark.parametrize("overlap", [False, True])
@pytest.mark.parametrize("prec", [sb.PREC_BF16, sb.PREC_TF32])
@pytest.mark.parametrize("d,K,n", [(1000, 8, 8200), (520, 8, 16384)])
def test_mixed_point_screen_same_bits_as_small_calls(d, K, n, prec, overlap):
    inst = _mixture(d, K, overlap)
    prob = sb.Problem(inst)
    x = _points(inst, n, d)
    ell, grad = sb.loglik(prob, x, prec)
    assert torch.equal(sb.loglik(prob, x, prec, want_grad=False), ell)
    for i0, m in ((0, 129), (n - 300, 300)):  # below the screen's line
        e, g = sb.loglik(prob, x[i0:i0 + m].contiguous(), prec)
        assert torch.equal(e, ell[i0:i0 + m]) and torch.equal(g, grad[i0:i0 + m])


@pytest.mark.parametrize("form", [2, 3])
@pytest.mark.parametrize("d,K,few,n_steps", [(22, 4, 181, 28), (3, 1, 1, 33), (130, 3, 257, 64), (64, 2, 40, 257)])
def test_ray_samples_do_not_depend_on_the_number_of_rays(d, K, few, n_steps, form):
    """Few rays take one pass per CTA, many up to eight."""
    prob = sb.Problem(_mixture(d, K, False))
    u = torch.randn(20000, d, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(d))
    u /= u.norm(dim=1, keepdim=True)
    ell = sb.ray_loglik_quad(prob, u, n_steps, form)
    assert torch.equal(sb.ray_loglik_quad(prob, u[:few].contiguous(), n_steps, form), ell[:few])
    assert torch.equal(sb.ray_loglik_quad(prob, u[-few:].contiguous(), n_steps, form), ell[-few:])


@pytest.mark.parametrize("d,K,n_modes", [(5, 2, 1), (33, 8, 6), (70, 3, 4), (40, 12, 5)])
def test_adjoint_of_a_mode_group_is_the_weighted_sum_of_its_modes(d, K, n_modes):
    """Modes are taken in groups of at most four: any number of them, one-hot or not, must
    give the log Z_k-weighted sum of the single-mode adjoints."""
    inst = _mixture(d, K, True)
    prob = sb.Problem(inst)
    rng = np.random.default_rng(d)
    modes = inst.mu[rng.integers(0, K, n_modes)] + 0.05 * rng.standard_normal((n_modes, d))
    modes[-1] += 30.0  # one component only: the one-hot branch
    logzk = rng.standard_normal(n_modes)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    dmu, dL = sb.evidence_backward(prob, t(modes), t(logzk), n_modes, 0.7)
    pi = np.exp(logzk - logzk.max())
    pi /= pi.sum()
    smu, sL = torch.zeros_like(dmu), torch.zeros_like(dL)
    for m in range(n_modes):
        a, b = sb.evidence_backward(prob, t(modes[m:m + 1]), t(logzk[m:m + 1]), 1, 0.7)
        smu += pi[m] * a
        sL += pi[m] * b
    ok = torch.isfinite(smu).all() and torch.isfinite(sL).all()
    assert bool(ok)
    for a, b in ((dmu, smu), (dL, sL)):
        assert float((a - b).abs().max()) <= 1e-13 * float(b.abs().max() + 1.0) * n_modes


@pytest.mark.parametrize("d,m", [(8, 64), (96, 40), (256, 33), (257, 5), (300, 64), (512, 20), (513, 3)])
def test_mixed_refinement_at_every_walker_width(d, m):
    """32, 64 or 128 threads a walker by d, histories longer than a warp's entries: walkers
    of a Gaussian reach its mean."""
    inst = make_instance(d, 1, 9 + d, s_range=(0.3, 1.0), mean_box=(-2, 2))
    prob = sb.Problem(inst)
    rng = np.random.default_rng(d)
    n = 70
    starts = torch.as_tensor(rng.uniform(-10, 10, (n, d)), device="cuda")
    cfg = sb.make_config(SolveConfig(n_rays=64, n_steps=64, n_starts=n, m=m, prec=sb.PREC_TF32))
    out = sb.refine(prob, cfg, starts)
    assert bool((out.status != sb.NONFINITE).all()) and bool((out.status != sb.MAXITER).all())
    err = (out.x - torch.as_tensor(inst.mu[0], device="cuda")).abs().amax(1)
    assert float(err.max()) < 2e-2
    lmax, _ = oracle.loglik(inst, inst.mu[0], want_grad=True)
    assert float((out.ell - lmax).abs().max()) < 1e-2 * (1 + abs(lmax))
