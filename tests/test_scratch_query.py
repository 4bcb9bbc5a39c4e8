"""Workspace queries hold what the call uses (host only; no GPU)."""
import ctypes as C

import pytest

import paper_2601_19957_gb300 as sb
from paper_2601_19957_gb300 import build as sbbuild


@pytest.fixture(scope="module", autouse=True)
def built():
    sbbuild.build()


@pytest.mark.parametrize("prec", [sb.PREC_TF32, sb.PREC_BF16])
@pytest.mark.parametrize("d,K,n", [(1024, 8, 16384), (300, 3, 1000), (7, 64, 129)])
def test_mixed_likelihood_asks_for_no_copy_of_its_results(d, K, n, prec):
    """The operands, their two L_k copies and what comes per row and component; values and
    gradients go to the caller's arrays, so nothing else is n x d."""
    p = sb._Problem(d, K, 0x1000, 0x1000, 0x1000, 0x1000, 0x1000)
    e = 2 if prec == sb.PREC_BF16 else 4
    rows, blocks = (n + 127) // 128 * 128, (n + 127) // 128
    ldp, ldz, tiles = (d + 7) // 8 * 8, (d + 63) // 64 * 64, (d + 63) // 64
    operands = 2 * K * d * ldp * e + K * rows * (ldp + ldz) * e
    per_row = rows * K * 4 * (tiles + 2) + 3 * rows * 4 + 2 * blocks * K * 4
    scratch = 2 * rows * d * 4  # the autotuner's and the skip bounds'
    small = K * d * 4 + d * 4 + K * 12 + (2 * d + 3) * 8
    query = int(sb.lib().sb_loglik_workspace_bytes(C.byref(p), prec, n))
    assert query <= operands + per_row + scratch + small + 256 * 24
