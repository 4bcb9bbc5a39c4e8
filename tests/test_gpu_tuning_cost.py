"""The tile autotuner's first call of a shape: a few launches where the widths differ."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2601_19957_gb300 as sb
from paper_2601_19957_gb300.instances import Instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [sb.PREC_BF16, sb.PREC_TF32])
def test_first_call_of_a_shape_launches_few_timings(prec, monkeypatch):
    """d = 960, three widths, 64 columns far behind: three pairs of GEMMs each, and at most five
    more for each of the other two when they tie."""
    monkeypatch.delenv("SB_TUNE", raising=False)
    d, K, n = 960, 5, 8192
    inst = Instance(d, K, np.full(K, -np.log(K)), np.zeros((K, d)), np.repeat(np.eye(d)[None], K, 0), np.full(d, -10.0),
                    np.full(d, 10.0))
    prob = sb.Problem(inst)
    x = torch.zeros(n, d, dtype=torch.float64, device="cuda")
    assert sb.lib().sb_tuned_tile(d, K, prec) == 0  # a shape of this test only
    count = sb.lib().sb_launch_count
    count.restype = C.c_int64
    a = count()
    sb.loglik(prob, x, prec)
    b = count()
    sb.loglik(prob, x, prec)
    tuning = (b - a) - (count() - b)
    assert sb.lib().sb_tuned_tile(d, K, prec) in (128, 256)
    assert 0 < tuning <= 2 * (3 * 3 + 2 * 5)
