"""Exit lengths of the rays from the box centre where half-widths lie outside FP32's range:
the tensor-core forms decide most of them by FP32 quotients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2601_19957_gb300 as sb
import tc_bound
from paper_2601_19957_gb300.instances import SolveConfig, make_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [2, 3])
@pytest.mark.parametrize("halves", [
    {5: 1e31},                 # one side far beyond the others
    {0: 1e31, 63: 3e40},       # beyond FP32 itself
    {17: 1e-31},               # one side below every other: it sets every exit
    {17: 1e-31, 40: 1e31},
    {17: 1e-31, 18: 1e-31},    # two of them in one lane
    {i: 1e31 for i in range(64)},
])
def test_exit_lengths_with_half_widths_outside_fp32(halves, form):
    d, K, n_rays, n_steps = 64, 3, 200, 16
    inst = make_instance(d, K, 700 + d, s_range=(0.05, 0.5), mean_box=(-6, 6), sep=8.0)
    for i, h in halves.items():
        inst.lo[i], inst.hi[i] = -h, h
    all_wide = len(halves) == d
    cfg = SolveConfig(n_rays=n_rays, n_steps=n_steps, n_starts=1, seed=d)
    u, te, ref = oracle.ray_loglik(inst, cfg)
    ell = sb.ray_loglik_quad(sb.Problem(inst), torch.as_tensor(u, device="cuda"), n_steps, form=form).cpu().numpy()
    half = 0.5 * (inst.hi - inst.lo)
    assert np.array_equal(te, (half / np.abs(u)).min(1))
    if all_wide:  # l about -1e64: relative
        assert np.allclose(ell, ref, rtol=1e-5, atol=0)
        return
    tau = (np.arange(1, n_steps + 1) / n_steps)[None, :] * te[:, None]
    X = (tau[:, :, None] * u[:, None, :]).reshape(-1, d)
    tc_bound.check_ray_samples(inst, X, (ell - ref).reshape(-1), {2: sb.PREC_BF16, 3: sb.PREC_TF32}[form])


@pytest.mark.parametrize("form", [2, 3])
def test_exit_lengths_of_axis_and_tied_directions(form):
    """One coordinate alone, all coordinates equal, two nearly equal: the same samples as FP64."""
    d, n_steps = 64, 8
    inst = make_instance(d, 2, 11, s_range=(0.3, 0.5), mean_box=(-6, 6), sep=8.0)
    inst.hi[3], inst.lo[3] = 1e31, -1e31
    u = np.zeros((6, d))
    u[0, 0] = u[1, 63] = 1.0
    u[2] = 1.0 / np.sqrt(d)
    u[3, 10] = u[3, 42] = np.sqrt(0.5)
    u[4, 10], u[4, 42] = np.sqrt(0.5), np.nextafter(np.sqrt(0.5), 1)
    u[5, 3], u[5, 4] = 0.6, 0.8
    t = torch.as_tensor(u, device="cuda")
    prob = sb.Problem(inst)
    want = sb.ray_loglik_quad(prob, t, n_steps, form=0).cpu().numpy()
    got = sb.ray_loglik_quad(prob, t, n_steps, form=form).cpu().numpy()
    X = ((np.arange(1, n_steps + 1) / n_steps)[None, :, None] * (10.0 / np.abs(np.where(np.arange(d) == 3, 0, u)).max(1))[:, None, None]
         * u[:, None, :]).reshape(-1, d)
    tc_bound.check_ray_samples(inst, X, (got - want).reshape(-1), {2: sb.PREC_BF16, 3: sb.PREC_TF32}[form])
