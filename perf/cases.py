"""The calls a user of this library makes, as timed cases.

Each kind of case is one public entry point over the range of sizes and options
it is used with: the likelihood on its own (a single point up to a full set of
walkers, FP64 / TF32 / BF16, with and without the gradient), the ray likelihood,
the preprocessing probe, the Laplace stage, the adjoint, and whole evidence
solves (one small problem, a mixture in FP64, the large mixed-precision mixture,
and a batch). Mixtures are those of `instances.make_instance` (Haar-rotated
covariances, log-uniform scales, Dirichlet weights, separated means, prior
[-10, 10]^d), drawn here on the GPU with torch so that preparing one is quick.
"""
import ctypes
import math

import torch

import paper_2601_19957_gb300 as sb
from paper_2601_19957_gb300.instances import SolveConfig

F64 = torch.float64
PREC = {"fp64": sb.PREC_FP64, "tf32": sb.PREC_TF32, "bf16": sb.PREC_BF16}
PRIOR = 10.0  # prior box [-PRIOR, PRIOR]^d


def listed():
    return [
        # l and grad l at one point of a mid-size mixture: an external sampler's or
        # optimiser's step through the FP64 likelihood, the smallest call there is
        {"name": "loglik_fp64_point", "kind": "loglik", "prec": "fp64", "d": 64, "K": 4, "n": 1, "grad": True},
        # the plain FP64 likelihood and gradient of a set of walkers
        {"name": "loglik_fp64_walkers", "kind": "loglik", "prec": "fp64", "d": 256, "K": 4, "n": 4096, "grad": True},
        # the mixed-precision likelihood and gradient at the size of the large solve's walkers
        {"name": "loglik_bf16_walkers", "kind": "loglik", "prec": "bf16", "d": 1024, "K": 8, "n": 16384, "grad": True},
        # values only at ragged sizes (nothing a multiple of a tile): scoring given points
        {"name": "loglik_tf32_values_ragged", "kind": "loglik", "prec": "tf32", "d": 300, "K": 3, "n": 5003,
         "grad": False},
        # discovery's coarse pass on its own: l at every sample of the sunburst rays
        {"name": "rays_bf16", "kind": "rays", "form": 2, "d": 1024, "K": 8, "n_rays": 16384, "n_steps": 64},
        # preprocessing of a large mixture with a few flat and soft coordinates
        {"name": "precheck_large", "kind": "precheck", "d": 1024, "K": 8},
        # Newton polish, Hessian, Cholesky and log Z of refined walkers; the components
        # overlap, so the Hessians are full sums
        {"name": "laplace_overlapping", "kind": "laplace", "d": 512, "K": 4, "n": 512},
        # the adjoint of log Z at the modes of an overlapping mixture (a training step's backward)
        {"name": "backward_overlapping", "kind": "backward", "d": 512, "K": 4, "overlap": True},
        # sunburst, L-BFGS and Laplace of one small correlated Gaussian in FP64: latency
        {"name": "evidence_fp64_small", "kind": "evidence", "prec": "fp64", "d": 8, "K": 1, "n_rays": 256,
         "n_steps": 64, "n_starts": 64, "m": 10, "chisao": False},
        # the whole pipeline in FP64 on a mixture
        {"name": "evidence_fp64_mixture", "kind": "evidence", "prec": "fp64", "d": 64, "K": 4, "n_rays": 1024,
         "n_steps": 128, "n_starts": 4096, "m": 10, "chisao": True},
        # the headline solve: the whole pipeline in BF16 at d = 1024
        {"name": "evidence_bf16_large", "kind": "evidence", "prec": "bf16", "d": 1024, "K": 8, "n_rays": 16384,
         "n_steps": 64, "n_starts": 16384, "m": 20, "chisao": True},
        # many uneven problems in one call
        {"name": "batch_tf32", "kind": "batch", "prec": "tf32", "P": 64, "d_max": 512, "K_max": 4, "n_rays": 512,
         "n_steps": 64, "n_starts": 512, "m": 10, "workers": 16},
    ]


def _logint(rng, lo, hi):
    """An integer of [lo, hi], uniform over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["loglik_fp64", "loglik_fp64", "loglik_mixed", "loglik_mixed", "rays", "precheck", "laplace",
                       "backward", "evidence_small", "evidence_fp64", "evidence_mixed", "batch"])
    if kind == "loglik_fp64":
        d, K = _logint(rng, 1, 512), rng.randint(1, 8)
        n = _logint(rng, 1, max(1, min(16384, int(2.5e8 / (K * d * (d + 1))))))
        return {"kind": "loglik", "prec": "fp64", "d": d, "K": K, "n": n, "grad": rng.random() < 0.6}
    if kind == "loglik_mixed":
        return {"kind": "loglik", "prec": rng.choice(["tf32", "bf16"]), "d": _logint(rng, 8, 1024),
                "K": rng.randint(1, 8), "n": _logint(rng, 64, 16384), "grad": rng.random() < 0.6}
    if kind == "rays":
        return {"kind": "rays", "form": rng.choice([2, 3]), "d": _logint(rng, 8, 1024), "K": rng.randint(1, 8),
                "n_rays": _logint(rng, 128, 16384), "n_steps": rng.randint(16, 64)}
    if kind == "precheck":
        return {"kind": "precheck", "d": _logint(rng, 2, 1024), "K": rng.randint(1, 8)}
    if kind == "laplace":
        return {"kind": "laplace", "d": _logint(rng, 8, 512), "K": rng.randint(1, 4), "n": _logint(rng, 16, 512)}
    if kind == "backward":
        return {"kind": "backward", "d": _logint(rng, 8, 512), "K": rng.randint(1, 4), "overlap": rng.random() < 0.6}
    if kind == "evidence_small":
        return {"kind": "evidence", "prec": "fp64", "d": _logint(rng, 8, 32), "K": 1, "n_rays": _logint(rng, 64, 512),
                "n_steps": rng.choice([32, 50, 64]), "n_starts": _logint(rng, 16, 256), "m": rng.choice([5, 10]),
                "chisao": False}
    if kind == "evidence_fp64":
        return {"kind": "evidence", "prec": "fp64", "d": rng.randint(24, 64), "K": rng.randint(1, 4), "n_rays": 1024,
                "n_steps": 128, "n_starts": rng.randint(1500, 4096), "m": 10, "chisao": True}
    if kind == "evidence_mixed":
        n = _logint(rng, 2048, 8192)
        return {"kind": "evidence", "prec": rng.choice(["tf32", "bf16"]), "d": _logint(rng, 96, 1024),
                "K": rng.randint(1, 4), "n_rays": n, "n_steps": 64, "n_starts": n, "m": rng.choice([10, 20]),
                "chisao": True}
    return {"kind": "batch", "prec": rng.choice(["tf32", "bf16"]), "P": rng.randint(8, 64),
            "d_max": rng.randint(64, 512), "K_max": rng.randint(1, 4), "n_rays": 512, "n_steps": 64, "n_starts": 512,
            "m": 10, "workers": rng.choice([8, 16])}


# --------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _cov_factor(d, g, s_lo, s_hi):
    """Lower Cholesky factor of P = Q diag(s^-2) Q^T, Q Haar, s log-uniform in [s_lo, s_hi]."""
    q, r = torch.linalg.qr(torch.randn(d, d, generator=g, dtype=F64, device="cuda"))
    q = q * torch.where(torch.diagonal(r) < 0, -1.0, 1.0)
    s = torch.exp(torch.rand(d, generator=g, dtype=F64, device="cuda") * math.log(s_hi / s_lo) + math.log(s_lo))
    p = (q / (s * s)) @ q.T
    return torch.linalg.cholesky(0.5 * (p + p.T))


def _weights(K, g):
    e = -torch.log(torch.rand(K, generator=g, dtype=F64, device="cuda"))
    return torch.log(e / e.sum())


def _mixture(d, K, g, s_lo=0.05, s_hi=0.5, half=6.0, sep=8.0):
    """A separated mixture as (log_w, mu, L, lo, hi); pairs of means more than sep * s_hi apart
    (no such rule below d = 8, where the box has no room for many of them)."""
    sep = sep if d >= 8 else 0.0
    L = torch.stack([_cov_factor(d, g, s_lo, s_hi) for _ in range(K)])
    mus = []
    while len(mus) < K:
        cand = (torch.rand(64, d, generator=g, dtype=F64, device="cuda") * 2 - 1) * half
        for c in cand:
            if len(mus) < K and all(float((c - m).norm()) > sep * s_hi for m in mus):
                mus.append(c)
    box = torch.full((d,), PRIOR, dtype=F64, device="cuda")
    return _weights(K, g), torch.stack(mus), L, -box, box


def _overlapping(d, K, g):
    """A tied-covariance mixture whose means lie 4.5 to 6 standard deviations apart along a
    line, so that every mode shares responsibility (of order 1e-5 to 1e-8) with its neighbours."""
    L = _cov_factor(d, g, 0.05, 0.5)
    v = torch.randn(1, d, generator=g, dtype=F64, device="cuda")
    v = v / v.norm()
    r = 4.5 + 1.5 * torch.rand(K, 1, generator=g, dtype=F64, device="cuda")
    steps = torch.linalg.solve_triangular(L.T, (v * r).T, upper=True).T
    c = torch.rand(d, generator=g, dtype=F64, device="cuda") * 2 - 1
    mu = c + torch.cumsum(steps, 0)
    w = 0.2 + 0.8 * torch.rand(K, generator=g, dtype=F64, device="cuda")
    box = torch.full((d,), PRIOR, dtype=F64, device="cuda")
    return torch.log(w / w.sum()), mu, L.expand(K, d, d).contiguous(), -box, box


def _consts(log_w, L):
    d = L.shape[-1]
    return log_w - 0.5 * d * math.log(2 * math.pi) + torch.log(torch.diagonal(L, dim1=-2, dim2=-1)).sum(-1)


def _terms(p, x):
    """e_k(x) [n][K] and z_k(x) [K][n][d] in FP64."""
    log_w, mu, L, _, _ = p
    z = torch.stack([(x - mu[k]) @ L[k] for k in range(L.shape[0])])
    return (_consts(log_w, L)[:, None] - 0.5 * (z * z).sum(-1)).T, z


def _loglik_ref(p, x, grad):
    e, z = _terms(p, x)
    ell = torch.logsumexp(e, 1)
    if not grad:
        return ell
    r = torch.exp(e - ell[:, None])
    g = torch.zeros_like(x)
    for k in range(z.shape[0]):
        g -= (r[:, k, None] * z[k]) @ p[2][k].T
    return ell, g


def _hessian(p, x):
    """-hess l at one point, with l and grad l (differentiable)."""
    log_w, mu, L, _, _ = p
    dl = x - mu
    z = torch.einsum("kij,ki->kj", L, dl)
    e = _consts(log_w, L) - 0.5 * (z * z).sum(-1)
    ell = torch.logsumexp(e, 0)
    r = torch.exp(e - ell)
    g = -torch.einsum("kij,kj->ki", L, z)
    gbar = (r[:, None] * g).sum(0)
    H = torch.einsum("k,kij,klj->il", r, L, L) - torch.einsum("k,ki,kl->il", r, g, g) + torch.outer(gbar, gbar)
    return ell, gbar, H


def _modes(p):
    """The modes next to the means (Newton from each mean), their l and log Z_k, by decreasing l."""
    out = []
    d = p[1].shape[1]
    for k in range(p[1].shape[0]):
        x = p[1][k].clone()
        for _ in range(6):
            _, g, H = _hessian(p, x)
            x = x + torch.cholesky_solve(g[:, None], torch.linalg.cholesky(H))[:, 0]
        ell, _, H = _hessian(p, x)
        C = torch.linalg.cholesky(H)
        out.append((x, ell, ell + 0.5 * d * math.log(2 * math.pi) - torch.log(torch.diagonal(C)).sum()))
    out.sort(key=lambda t: -float(t[1]))
    return tuple(torch.stack([o[i] for o in out]) for i in range(3))


def _points(p, n, g):
    """n points as walkers and scored samples see them: around the components at |z_k| from
    0.1 to 100, a tenth of them uniform in the box."""
    log_w, mu, L, lo, hi = p
    K, d = mu.shape
    x = torch.empty(n, d, dtype=F64, device="cuda")
    lab = torch.randint(K, (n,), generator=g, device="cuda")
    rad = torch.exp(torch.rand(n, 1, generator=g, dtype=F64, device="cuda") * math.log(1000.0) + math.log(0.1))
    z = torch.randn(n, d, generator=g, dtype=F64, device="cuda")
    z = z * (rad / z.norm(dim=1, keepdim=True))
    for k in range(K):
        sel = torch.nonzero(lab == k).flatten()
        x[sel] = mu[k] + torch.linalg.solve_triangular(L[k].T, z[sel].T, upper=True).T
    far = torch.rand(n, 1, generator=g, device="cuda") < 0.1
    u = torch.rand(n, d, generator=g, dtype=F64, device="cuda") * 2 - 1
    return torch.where(far, u * PRIOR, x).clamp(-PRIOR, PRIOR).contiguous()


def _precheck_problem(case, g):
    """A separated mixture whose last coordinates are flat (a tiny precision) or soft."""
    d, K = case["d"], case["K"]
    nf = d // 32
    ns = d // 32
    da = d - nf - ns
    log_w, mu_a, L_a, lo, hi = _mixture(da, K, g)
    mu = torch.zeros(K, d, dtype=F64, device="cuda")
    mu[:, :da] = mu_a
    L = torch.zeros(K, d, d, dtype=F64, device="cuda")
    L[:, :da, :da] = L_a
    diag = torch.empty(nf + ns, dtype=F64, device="cuda")
    diag[:nf] = 1e-5 * (1 + torch.rand(nf, generator=g, dtype=F64, device="cuda"))
    diag[nf:] = 0.02 * (1 + torch.rand(ns, generator=g, dtype=F64, device="cuda"))
    idx = torch.arange(da, d, device="cuda")
    L[:, idx, idx] = diag
    box = torch.full((d,), PRIOR, dtype=F64, device="cuda")
    return log_w, mu, L, -box, box


def _evidence_problem(case, g):
    if case["K"] == 1:
        return _mixture(case["d"], 1, g, 0.1, 1.0, 2.0)
    return _mixture(case["d"], case["K"], g, sep=10.0 if case["d"] >= 512 else 8.0)


def _batch_problems(case, seed):
    g = _gen(seed)
    rng = torch.Generator()
    rng.manual_seed(int(seed) & 0x7FFFFFFF)
    ds = (torch.randint(1, case["d_max"] // 16 + 1, (case["P"],), generator=rng) * 16).tolist()
    Ks = torch.randint(1, case["K_max"] + 1, (case["P"],), generator=rng).tolist()
    return [_mixture(d, K, g) for d, K in zip(ds, Ks)]


def _laplace_inputs(case, g):
    """Refined walkers as a mixed-precision L-BFGS leaves them: scattered about the modes at
    about 1e-4 of a standard deviation."""
    p = _overlapping(case["d"], case["K"], g)
    n, d, K = case["n"], case["d"], case["K"]
    modes, _, _ = _modes(p)
    lab = torch.arange(n, device="cuda") % K
    z = torch.randn(n, d, generator=g, dtype=F64, device="cuda") * (1e-4 / math.sqrt(d))
    x = modes[lab] + torch.linalg.solve_triangular(p[2][0].T, z.T, upper=True).T
    return p, x.contiguous()


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "batch":
        ps = _batch_problems(case, seed)
        st["probs"] = [sb.TensorProblem(*p) for p in ps]
        st["cfg"] = sb.make_config(SolveConfig(n_rays=case["n_rays"], n_steps=case["n_steps"],
                                               n_starts=case["n_starts"], m=case["m"], seed=seed,
                                               prec=PREC[case["prec"]]))
        st["cc"] = sb.make_chisao_config(n_osc=3, anti_alpha=0.1)
        st["ws"] = sb.batched_workspace(st["probs"], st["cfg"], case["workers"], chisao=True)
        st["out"] = (torch.empty(case["P"], dtype=F64, device="cuda"),
                     torch.empty(case["P"], dtype=torch.int32, device="cuda"))
        return st
    if kind == "loglik":
        p = _mixture(case["d"], case["K"], g)
        st["x"] = _points(p, case["n"], g)
        st["prob"] = sb.TensorProblem(*p)
        st["ws"] = sb.Workspace(sb.lib().sb_loglik_workspace_bytes(ctypes.byref(st["prob"].s), PREC[case["prec"]],
                                                                   case["n"]))
    elif kind == "rays":
        p = _mixture(case["d"], case["K"], g)
        u = torch.randn(case["n_rays"], case["d"], generator=g, dtype=F64, device="cuda")
        st["u"] = (u / u.norm(dim=1, keepdim=True)).contiguous()
        st["prob"] = sb.TensorProblem(*p)
    elif kind == "precheck":
        st["prob"] = sb.TensorProblem(*_precheck_problem(case, g))
    elif kind == "laplace":
        p, st["x"] = _laplace_inputs(case, g)
        st["ell"] = _loglik_ref(p, st["x"], False)
        st["prob"] = sb.TensorProblem(*p)
        st["cfg"] = sb.make_config(SolveConfig(n_rays=64, n_starts=case["n"], cand_cap=64, seed=seed))
        st["ws"] = sb.workspace(st["prob"], st["cfg"])
    elif kind == "backward":
        p = _overlapping(case["d"], case["K"], g) if case["overlap"] else _mixture(case["d"], case["K"], g)
        st["modes"], _, st["logZk"] = _modes(p)
        st["prob"] = sb.TensorProblem(*p)
    else:
        st["prob"] = sb.TensorProblem(*_evidence_problem(case, g))
        st["cfg"] = sb.make_config(SolveConfig(n_rays=case["n_rays"], n_steps=case["n_steps"],
                                               n_starts=case["n_starts"], m=case["m"], seed=seed,
                                               prec=PREC[case["prec"]]))
        st["cc"] = sb.make_chisao_config(n_osc=3, anti_alpha=0.1)
        st["ws"] = (sb.chisao_workspace if case["chisao"] else sb.workspace)(st["prob"], st["cfg"])
        st["out"] = sb.EvidenceBuffers(case["d"], st["cfg"].cand_cap)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "loglik":
        return sb.loglik(st["prob"], st["x"], PREC[case["prec"]], case["grad"], ws=st["ws"])
    if kind == "rays":
        return sb.ray_loglik_quad(st["prob"], st["u"], case["n_steps"], case["form"])
    if kind == "precheck":
        o = sb.precheck(st["prob"])
        return o.s, o.cls, o.log_int, o.log_vol, o.n_active
    if kind == "laplace":
        o = sb.laplace(st["prob"], st["cfg"], st["x"], st["ell"], ws=st["ws"])
        return o.logZ, o.modes, o.logZk, o.ell, o.n_modes
    if kind == "backward":
        return sb.evidence_backward(st["prob"], st["modes"], st["logZk"], st["modes"].shape[0])
    if kind == "batch":
        return sb.evidence_batched(st["probs"], st["cfg"], case["workers"], ws=st["ws"], out=st["out"], cc=st["cc"])
    if case["chisao"]:
        o = sb.evidence_chisao(st["prob"], st["cfg"], st["cc"], ws=st["ws"], out=st["out"])
    else:
        o = sb.evidence(st["prob"], st["cfg"], ws=st["ws"], out=st["out"])
    return o.logZ, o.modes, o.logZk, o.n_modes


def work(case):
    """Algorithmic bytes and flops of one pass. The triangle of every L_k is read once; a
    likelihood evaluation is K d (d + 1) flops, with its gradient twice that. Whole solves
    count a typical number of L-BFGS evaluations per start (the sunburst-only small solve
    about 30, a ChiSao solve about 200)."""
    kind = case["kind"]
    if kind == "batch":
        d, K = case["d_max"] / 2, case["K_max"] / 2 + 0.5
        tri = K * d * (d + 1)
        ev = 200 * case["n_starts"] * 2 + case["n_rays"] * 1
        return {"bytes": case["P"] * (4 * tri + 16), "flops": case["P"] * ev * tri}
    d, K = case["d"], case["K"]
    tri = K * d * (d + 1)
    inp = 4.0 * tri + 8.0 * K * (d + 1) + 16.0 * d
    if kind == "loglik":
        g = 2 if case["grad"] else 1
        return {"bytes": inp + 8.0 * case["n"] * (d * g + 1), "flops": float(case["n"]) * tri * g}
    if kind == "rays":
        return {"bytes": inp + 8.0 * case["n_rays"] * (d + case["n_steps"]), "flops": float(case["n_rays"]) * tri}
    if kind == "precheck":
        return {"bytes": inp + 9.0 * d, "flops": 3.0 * tri}
    if kind == "laplace":
        # l, grad l, the assembled Hessian and its factor at the K modes before and after one Newton step
        return {"bytes": inp + 8.0 * case["n"] * (d + 1) + 8.0 * K * d,
                "flops": 2.0 * K * (2.0 * tri + d ** 3 / 3.0) + K * d ** 3 / 3.0}
    if kind == "backward":
        # per mode: H assembled and factored, W applied to every active L_k
        f = K * (d ** 3 / 3.0 + (K * 2.0 * d ** 3 if case["overlap"] else 0.0)) + 8.0 * K * tri
        return {"bytes": inp + 4.0 * tri + 8.0 * K * d * 2, "flops": f}
    per = 200 if case["chisao"] else 30
    ev = per * case["n_starts"] * 2 + case["n_rays"]
    return {"bytes": inp + 8.0 * (K * (d + 1) + 1), "flops": float(ev) * tri}


# --------------------------------------------------------------------------- 64-bit values
def _backward_ref(p, modes, logZk):
    """d log Z / d (mu, L) with the implicit shift of the modes, by autograd in FP64: at a mode
    d log Z_m = d [l - log det H / 2 - v . grad l / 2], v = H^-1 grad_x log det H held fixed."""
    log_w, mu, L, lo, hi = p
    mu = mu.clone().requires_grad_(True)
    L = L.clone().requires_grad_(True)
    pi = torch.softmax(logZk, 0)
    gm, gL = torch.zeros_like(mu), torch.zeros_like(L)
    for m in range(modes.shape[0]):
        x = modes[m].clone().requires_grad_(True)
        _, _, H = _hessian((log_w, mu.detach(), L.detach(), lo, hi), x)
        C = torch.linalg.cholesky(H)
        t, = torch.autograd.grad(2 * torch.log(torch.diagonal(C)).sum(), x)
        v = torch.cholesky_solve(t[:, None], C.detach())[:, 0]
        ell, gbar, H = _hessian((log_w, mu, L, lo, hi), modes[m])
        C = torch.linalg.cholesky(H)
        f = ell - torch.log(torch.diagonal(C)).sum() - 0.5 * (v * gbar).sum()
        a, b = torch.autograd.grad(pi[m] * f, (mu, L))
        gm += a
        gL += b
    return gm, torch.tril(gL)


def _precheck_ref(p):
    log_w, mu, L, lo, hi = p
    c, half = 0.5 * (lo + hi), 0.5 * (hi - lo)
    e, z = _terms(p, c[None])
    r = e[0] - torch.logsumexp(e[0], 0)
    dot = torch.einsum("kij,kj->ki", L, z[:, 0])
    nrm = (L * L).sum(-1)
    s = sum(torch.logsumexp(r[:, None] - t * dot - 0.5 * t * t * nrm, 0).abs() for t in (half, -half))
    v = torch.sort(s).values
    d = s.shape[0]
    med = v[d // 2] if d % 2 else 0.5 * (v[d // 2 - 1] + v[d // 2])
    flat = s < 1e-6 * med
    soft = ~flat & (s < 1e-3 * v[-1])
    lw = torch.log(2 * half)
    li = lw[flat].sum() + (0.5 * math.log(2 * math.pi) + torch.log(half / torch.sqrt(s)))[soft].sum()
    cls = flat.to(torch.int8) + 2 * soft.to(torch.int8)
    return s, cls, float(li), float(lw[flat | soft].sum()), int((cls == 0).sum())


def _rays_ref(p, u, n_steps):
    log_w, mu, L, lo, hi = p
    c, half = 0.5 * (lo + hi), 0.5 * (hi - lo)
    texit = (half / u.abs()).min(1).values
    tau = texit[:, None] * torch.arange(1, n_steps + 1, dtype=F64, device="cuda") / n_steps
    a = _consts(log_w, L)
    e = []
    for k in range(L.shape[0]):
        z0 = (c - mu[k]) @ L[k]
        w = u @ L[k]
        e.append(a[k] - 0.5 * ((z0 * z0).sum() + 2 * tau * (w @ z0)[:, None] + tau * tau * (w * w).sum(1)[:, None]))
    return torch.logsumexp(torch.stack(e), 0)


def exact(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "loglik":
        p = _mixture(case["d"], case["K"], g)
        return _loglik_ref(p, _points(p, case["n"], g), case["grad"])
    if kind == "rays":
        p = _mixture(case["d"], case["K"], g)
        u = torch.randn(case["n_rays"], case["d"], generator=g, dtype=F64, device="cuda")
        return _rays_ref(p, u / u.norm(dim=1, keepdim=True), case["n_steps"])
    if kind == "precheck":
        return _precheck_ref(_precheck_problem(case, g))
    logV = case.get("d", 0) * math.log(2 * PRIOR)
    if kind == "laplace":
        p, _ = _laplace_inputs(case, g)
        x, ell, zk = _modes(p)
        return float(torch.logsumexp(zk, 0)) - logV, x, zk, ell, x.shape[0]
    if kind == "backward":
        p = _overlapping(case["d"], case["K"], g) if case["overlap"] else _mixture(case["d"], case["K"], g)
        x, _, zk = _modes(p)
        return _backward_ref(p, x, zk)
    if kind == "batch":
        ps = _batch_problems(case, seed)
        return (torch.tensor([-p[1].shape[1] * math.log(2 * PRIOR) for p in ps], dtype=F64, device="cuda"),
                torch.tensor([p[1].shape[0] for p in ps], dtype=torch.int32, device="cuda"))
    # separated mixtures: the modes are the means, log Z_k = log w_k, log Z = -log V
    p = _evidence_problem(case, g)
    order = torch.argsort(_consts(p[0], p[2]), descending=True)
    return -logV, p[1][order], p[0][order], case["K"]
