"""Shared-memory permissions of kernels belong to one device: the routes that serve every
device of a process ask before each launch, not once (read from the sources; no GPU)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_19957_gb300", "csrc")
# asked once per process: the tensor-core GEMMs, the FP32 step and ChiSao's bases
ONCE = {"k_tc_gemm", "k_lbfgs_cta", "k_cs_bases"}


def _requests():
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"(?:cudaFuncSetAttribute|allow_smem)\(\s*(k\w*)", text):
            statement = re.split(r"[;{}]", text[:m.start()])[-1]
            # a lambda of call_once opens at most a few statements earlier
            before = text[max(0, m.start() - 400):m.start()]
            once = re.search(r"\bstatic\b", statement) or (
                "call_once" in before and before[before.rindex("call_once"):].count("});") == 0)
            yield name, m.group(1), bool(once)


def test_the_scan_sees_the_requests():
    seen = {k for _, k, _ in _requests()}
    assert ONCE | {"k_ggemm_f64_grouped", "k_ray_bucket", "k_tc_lse", "k_precision", "k_adj_solve"} <= seen
    assert {k for _, k, once in _requests() if once} >= ONCE


@pytest.mark.parametrize("kernel", ["k_ggemm_f64_grouped", "k_ray_bucket", "k_tc_lse", "k_precision", "k_adj_solve"])
def test_permission_is_asked_before_each_launch(kernel):
    assert [once for _, k, once in _requests() if k == kernel] == [False]


def test_no_other_kernel_is_asked_for_once():
    assert {k for _, k, once in _requests() if once} == ONCE
