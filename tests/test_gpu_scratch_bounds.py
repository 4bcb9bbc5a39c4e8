"""Calls on a workspace of exactly the queried size: nothing past it is written."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2601_19957_gb300 as sb
from paper_2601_19957_gb300.instances import make_instance

pytestmark = pytest.mark.gpu

GUARD = 64 * 1024  # more than any of the constants written per coordinate, d <= 1024


@pytest.mark.parametrize("prec", [sb.PREC_FP64, sb.PREC_TF32, sb.PREC_BF16])
@pytest.mark.parametrize("n,K", [(1, 1), (1, 2), (3, 1)])
@pytest.mark.parametrize("d", [1, 31, 64, 129, 512, 1024])
def test_loglik_stays_inside_its_workspace(d, n, K, prec):
    inst = make_instance(d, K, 5 + d, s_range=(0.2, 0.5), mean_box=(-6, 6))
    prob = sb.Problem(inst)
    x = torch.as_tensor(inst.mu[np.arange(n) % K] + 0.1, device="cuda")
    need = int(sb.lib().sb_loglik_workspace_bytes(C.byref(prob.s), prec, n))
    buf = torch.full((need + GUARD,), 0x5A, dtype=torch.uint8, device="cuda")
    ell = torch.empty(n, dtype=torch.float64, device="cuda")
    grad = torch.empty_like(x)
    code = sb.lib().sb_loglik(C.byref(prob.s), C.c_int32(prec), sb._ptr(x), C.c_int32(n), sb._ptr(ell), sb._ptr(grad),
                              C.c_void_p(buf.data_ptr()), C.c_size_t(need), sb._stream())
    assert code == sb.SB_OK
    assert bool((buf[need:] == 0x5A).all())
    if prec == sb.PREC_FP64:
        want = np.array([oracle.loglik(inst, p) for p in x.cpu().numpy()])
        assert np.allclose(ell.cpu().numpy(), want, rtol=1e-12, atol=1e-12)
    # the checks of the box stay: an empty side is reported
    inst.hi[d - 1] = inst.lo[d - 1]
    bad = sb.Problem(inst)
    sb.lib().sb_loglik(C.byref(bad.s), C.c_int32(prec), sb._ptr(x), C.c_int32(n), sb._ptr(ell), None,
                       C.c_void_p(buf.data_ptr()), C.c_size_t(need), sb._stream())
    assert sb.lib().sb_check(C.c_void_p(buf.data_ptr()), C.c_size_t(need), sb._stream()) == sb.SB_ERR_INVALID_ARG


def _backward(prob, modes, logzk, nbytes):
    """sb_evidence_backward on exactly nbytes with a guard behind them."""
    buf = torch.full((nbytes + GUARD,), 0x5A, dtype=torch.uint8, device="cuda")
    dmu, dL = torch.empty_like(prob.mu), torch.empty_like(prob.L)
    code = sb.lib().sb_evidence_backward(C.addressof(prob.s), sb._ptr(modes), sb._ptr(logzk), modes.shape[0], 0.7,
                                         sb._ptr(dmu), sb._ptr(dL), C.c_void_p(buf.data_ptr()), nbytes, sb._stream())
    assert bool((buf[nbytes:] == 0x5A).all())
    return code, dmu, dL


def _one_mode_bytes(d, K):
    """Room for one mode with its own C^-1 L_k beside P_k: P_k and M_k [K][d][d], H, the
    vectors of a mode and the constants, each on a multiple of 256 bytes."""
    tiles, up = (d + 63) // 64, lambda n, s: (n * s + 255) // 256 * 256
    doubles = [32, K, d, d, 1, 1, K * d * d, d * d, K * d * d, K * d, K, K * tiles, d, 1, K * d, d * (K + 1), d, d, K,
               K * d, d, K, K * d, d, 1024]
    return sum(up(n, 8) for n in doubles) + sum(up(n, 4) for n in (1, 1, 1, 2))


@pytest.mark.parametrize("d,K,n_modes", [(1, 1, 1), (2, 64, 3), (5, 2, 5), (33, 8, 6), (64, 12, 5), (129, 3, 4),
                                         (256, 2, 7)])
def test_adjoint_results_do_not_depend_on_the_workspace(d, K, n_modes):
    """From the queried size (up to four modes together) down to one mode's."""
    inst = make_instance(d, K, 70 + d + K, s_range=(0.2, 0.5), mean_box=(-0.2, 0.2), sep=0.0)
    prob = sb.Problem(inst)
    rng = np.random.default_rng(d)
    modes = inst.mu[rng.integers(0, K, n_modes)] + 0.05 * rng.standard_normal((n_modes, d))
    if n_modes > 1:
        modes[-1] += 30.0  # a one-hot mode
    modes = torch.as_tensor(modes, device="cuda")
    logzk = torch.as_tensor(rng.standard_normal(n_modes), device="cuda")
    full = int(sb.lib().sb_evidence_backward_workspace_bytes(C.byref(prob.s)))
    code, dmu, dL = _backward(prob, modes, logzk, full)
    assert code == sb.SB_OK and bool(torch.isfinite(dmu).all()) and bool(torch.isfinite(dL).all())
    one = min(full, _one_mode_bytes(d, K))
    for nbytes in {one, (one + full) // 2 // 256 * 256, max(full - 256, one)}:
        code, a, b = _backward(prob, modes, logzk, nbytes)
        assert code == sb.SB_OK
        assert torch.equal(a, dmu) and torch.equal(b, dL)
    assert _backward(prob, modes, logzk, 8 * (2 * K + 1) * d * d)[0] == sb.SB_ERR_WORKSPACE
