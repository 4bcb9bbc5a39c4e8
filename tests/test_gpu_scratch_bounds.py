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
