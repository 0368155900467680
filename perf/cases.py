"""What the library is asked to do in use, as measurable cases.

Every case goes through the public entry points of `paper_1104_5497_gb300.nphc` (and
`autograd`) with the handles a user's program keeps: the system, the options, a result or
caller-owned endpoint arrays and their workspace.  `listed()` holds one case per use,
`draw()` more of the same ranges.

The kinds of case:
  solve      the whole method on one ring into a kept result, then its stationary points
             (read = "sps") or every certified complex solution (read = "solutions")
  batch      many disordered rings of mixed sizes solved together
  chunk      step by step on a sample of a large ring's paths: FP32 tracking, FP64
             continuation of the hand-offs, refinement and certification
  gradient   stationary points as a differentiable function of sigma, forward and backward
  adjoint    the couplings' gradient of a loss over given stationary points
  certify    points found by another method: refine, certify, deduplicate, classify
  quadratic  the whole method on a generic quadratic system
  endgame    the Cauchy endgame on a ring with positive-dimensional solution sets

Outputs are what a program takes from these calls: solutions, their classes and data.  A
solve's step and solve counts, alpha, beta and the residual of a converged point are left
out: the first depend on the rounding of every step, the others are rounding errors
themselves and have no digits to compare.  So are the numbers of diverged and failed paths
(one path to infinity may end as either); the certified ones are all there.  Arrays have
the shape of the buffers a program keeps for them (stationary points: a capacity by ring
size; solutions: one row per path), zero where there is nothing.  Angles are given modulo
2 pi, in [0, 2 pi) up to a guard of 1e-6, since those of collinear points are pi up to the
sign of a rounding error.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1104_5497_gb300 import autograd, inputs, nphc

CERTIFIED = (nphc.END_REAL, nphc.END_NONREAL, nphc.END_UNDECIDED)


def listed():
    return [
        # a small ring of the paper (sigma = 0.75; sigma = 0.0 below: U[0.5, 3] from the seed): latency
        dict(name="solve_n5", kind="solve", N=5, sigma=0.75, disorder=0.0, precision="mixed", tuned=False,
             read="sps"),
        # a disordered ring of ordinary size, all its complex solutions read back
        dict(name="solutions_n8", kind="solve", N=8, sigma=0.0, disorder=0.1, precision="mixed", tuned=False,
             read="solutions"),
        # the benchmark's ring: 262,144 paths, default options
        dict(name="solve_n10", kind="solve", N=10, sigma=0.0, disorder=0.0, precision="mixed", tuned=False,
             read="sps"),
        # the paper's N = 11 (1,048,576 paths), with the autotuner's corrector options
        dict(name="solve_n11", kind="solve", N=11, sigma=0.75, disorder=0.0, precision="mixed", tuned=True,
             read="sps"),
        # the plain FP64 mode
        dict(name="solve_n8_fp64", kind="solve", N=8, sigma=0.0, disorder=0.1, precision="fp64", tuned=False,
             read="sps"),
        # an ensemble of disordered rings, N = 6 .. 9, solved together
        dict(name="batch24", kind="batch", count=24, lo=6, hi=9),
        # a part of a ring too large to solve at once: N = 13 has 16.8 M paths
        dict(name="chunk_n13", kind="chunk", N=13, count=20011),
        # one step of fitting sigma to stationary-point data: forward and backward
        dict(name="gradient_n6", kind="gradient", N=6, disorder=0.1),
        # the backward pass alone, over as many points as the benchmark's ring has
        dict(name="adjoint_n10", kind="adjoint", N=10, count=1670),
        # certifying and classifying points that a random-start Newton search found
        dict(name="certify_n10", kind="certify", N=10, count=15013),
        # a dense random system of quadratics: 1,024 paths
        dict(name="quadratic_n10", kind="quadratic", n=10, terms=30),
        # singular endpoints of the ring with a positive-dimensional solution set
        dict(name="endgame_n4", kind="endgame", N=4, count=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "chunk", "gradient", "adjoint", "certify",
                       "quadratic", "endgame"])
    if kind == "solve":
        fp64 = rng.random() < 0.25
        N = rng.randint(5, 8 if fp64 else 10)
        # clean rings with N = 0 mod 4 have singular families: solved with disorder here
        disorder = round(rng.uniform(0.02, 0.2), 3) if N % 4 == 0 or rng.random() < 0.5 else 0.0
        return dict(kind=kind, N=N, sigma=0.0, disorder=disorder, precision="fp64" if fp64 else "mixed",
                    tuned=rng.random() < 0.5, read=rng.choice(["sps", "solutions"]) if N < 9 else "sps")
    if kind == "batch":
        lo = rng.randint(5, 8)
        return dict(kind=kind, count=_log_int(rng, 3, 24), lo=lo, hi=min(9, lo + rng.randint(0, 3)))
    if kind == "chunk":
        return dict(kind=kind, N=rng.randint(9, 13), count=_log_int(rng, 300, 20000))
    if kind == "gradient":
        return dict(kind=kind, N=rng.randint(5, 7), disorder=round(rng.uniform(0.02, 0.2), 3))
    if kind == "adjoint":
        return dict(kind=kind, N=rng.randint(4, 13), count=_log_int(rng, 6, 24830))
    if kind == "certify":
        return dict(kind=kind, N=rng.randint(5, 13), count=_log_int(rng, 100, 15000))
    if kind == "quadratic":
        n = rng.randint(3, 10)
        return dict(kind=kind, n=n, terms=rng.randint(n, 3 * n))
    return dict(kind=kind, N=rng.choice([4, 4, 5]), count=rng.randint(17, 64))


# ------------------------------------------------------------------ inputs --
def _ring(N, disorder, seed, sigma=0.0):
    """A ring with sigma ~ U[0.5, 3] (if 0), gamma on the unit circle and, with disorder, one
    normal draw per pair; its couplings d_ij^-sigma (1 + disorder g_ij)."""
    rng = np.random.default_rng(seed)
    drawn = float(rng.uniform(0.5, 3.0))
    sigma = sigma or drawn
    gamma = inputs.draw_gamma(rng)
    g = inputs.draw_pair_normals(rng, N) if disorder else np.zeros((N, N))
    return gamma, _couplings(N, sigma, g, disorder)


def _couplings(N, sigma, g, eps):
    i = np.arange(N)
    d = np.abs(i[:, None] - i[None, :])
    d = np.minimum(d, N - d)
    J = np.where(d > 0, np.maximum(d, 1).astype(float) ** -sigma, 0.0)
    return J * (1.0 + eps * g)


def _options(case, gamma):
    fp64 = case.get("precision") == "fp64"
    opts = nphc.options_default(gamma=gamma, precision=nphc.PREC_FP64 if fp64 else nphc.PREC_MIXED)
    if case.get("tuned"):   # what the autotuner picks on rings of these sizes
        opts.max_newton_fp32, opts.eps_fp32 = 2, 3e-5
    return opts


def _batch_instances(case, seed):
    """Disordered rings with sigma ~ U[0.5, 3], their sizes lo .. hi in turn."""
    sizes = [case["lo"] + i % (case["hi"] - case["lo"] + 1) for i in range(case["count"])]
    return [inputs.disordered_batch(1, seed + 1009 * i, n_lo=N, n_hi=N)[0] for i, N in enumerate(sizes)]


def _grad_hess(theta, J):
    """Gradient and Hessian of V at [count, M] angles (real or complex), theta_N = 0."""
    M = theta.shape[1]
    th = torch.cat([theta, torch.zeros_like(theta[:, :1])], 1)
    d = th[:, :, None] - th[:, None, :]
    g = (J * torch.sin(d)).sum(2)[:, :M]
    C = J * torch.cos(d)
    return g, torch.diag_embed(C.sum(2)[:, :M]) - C[:, :M, :M]


def _newton_angles(theta, J, iters):
    for _ in range(iters):
        g, H = _grad_hess(theta, J)
        step = torch.linalg.solve_ex(H, g.unsqueeze(2))[0].squeeze(2)
        size = step.abs().amax(1, keepdim=True)
        theta = theta - torch.nan_to_num(step * torch.clamp(1.0 / size, max=1.0))
    return theta


def _angles(J, count, seed, complex_part=0.0):
    """`count` stationary points (complex128 angles, theta_N = 0) by Newton's method from
    random starts; a `complex_part` of the starts are off the real torus.  Solutions repeat,
    as they do in a random-start search."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    Jc = torch.as_tensor(J, dtype=torch.complex128, device="cuda")
    M, found, have = len(J) - 1, [], 0
    while have < count:
        n = 2 * count + 64
        re = (torch.rand(n, M, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1) * math.pi
        im = torch.randn(n, M, generator=gen, device="cuda", dtype=torch.float64)
        off = torch.rand(n, 1, generator=gen, device="cuda") < complex_part
        th = _newton_angles(torch.complex(re, im * off * 0.7), Jc, 40)
        g, H = _grad_hess(th, Jc)
        scale = torch.linalg.matrix_norm(torch.nan_to_num(H))
        inv = torch.linalg.matrix_norm(torch.nan_to_num(torch.linalg.inv_ex(H)[0], nan=math.inf))
        good = (g.abs().amax(1) < 1e-11) & (scale * inv < 1e5) & (th.imag.abs().amax(1) < 4)
        found.append(th[good])
        have += int(good.sum())
    return torch.cat(found)[:count]


def _quadratic(case, seed):
    """A random system: z_i^2 plus `terms` random quadratic, linear and constant terms per
    equation; complex normal coefficients.  Returned as the term list of the entry point."""
    rng = np.random.default_rng(seed)
    n, k = case["n"], case["terms"]
    eq = np.repeat(np.arange(n), k + 1)
    va = rng.integers(-1, n, n * (k + 1))
    vb = rng.integers(-1, n, n * (k + 1))
    coef = (rng.standard_normal(len(eq)) + 1j * rng.standard_normal(len(eq))) / np.sqrt(2 * k)
    first = np.arange(n) * (k + 1)
    va[first] = vb[first] = np.arange(n)
    coef[first] = 1.0
    return eq, va, vb, coef, inputs.draw_gamma(rng)


# ------------------------------------------------------- prepare and run --
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "solve":
        gamma, J = _ring(case["N"], case["disorder"], seed, case["sigma"])
        s["system"] = nphc.System(case["N"], J=J)
        s["opts"] = _options(case, gamma)
        s["result"] = nphc.Result(s["system"])
    elif kind == "batch":
        inst = _batch_instances(case, seed)
        s["systems"] = [nphc.System(i.N, J=nphc.xy_couplings(i.N, i.sigma, i.g, i.eps)) for i in inst]
        s["opts"] = [nphc.options_default(gamma=i.gamma) for i in inst]
        s["batch"] = nphc.Batch(s["systems"])
    elif kind == "chunk":
        gamma, J = _ring(case["N"], 0.1, seed)
        s["system"] = system = nphc.System(case["N"], J=J)
        s["opts"] = nphc.options_default(gamma=gamma)
        paths = np.random.default_rng(seed).choice(system.npaths, case["count"], replace=False)
        s["ep"] = nphc.DeviceEndpoints.empty(system.n, np.sort(paths))
        s["ws"] = torch.empty(system.workspace_size(case["count"]), dtype=torch.uint8, device="cuda")
    elif kind == "gradient":
        rng = np.random.default_rng(seed)
        s["g"] = inputs.draw_pair_normals(rng, case["N"])
        s["gamma"] = inputs.draw_gamma(rng)
        s["value"] = torch.tensor(float(rng.uniform(0.5, 3.0)), dtype=torch.float64, requires_grad=True)
    elif kind == "adjoint":
        _, J = _ring(case["N"], 0.1, seed)
        s["system"] = nphc.System(case["N"], J=J)
        s["theta"], s["g_energy"], s["g_theta"] = _adjoint_inputs(case, J, seed)
    elif kind == "certify":
        gamma, J = _ring(case["N"], 0.1, seed)
        s["system"] = system = nphc.System(case["N"], J=J)
        s["opts"] = nphc.options_default(gamma=gamma)
        n, M = case["count"], case["N"] - 1
        z = _certify_points(case, J, seed)
        noise = torch.Generator(device="cuda").manual_seed(seed + 1)
        z = z * (1 + 1e-6 * torch.randn(z.shape, generator=noise, device="cuda", dtype=torch.complex128))
        s["z_re"], s["z_im"] = z.real.T.contiguous(), z.imag.T.contiguous()
        s["ep"] = nphc.DeviceEndpoints.empty(system.n, np.arange(n))
        s["ws"] = torch.empty(system.workspace_size(n), dtype=torch.uint8, device="cuda")
        f64 = dict(dtype=torch.float64, device="cuda")
        s["theta"] = torch.zeros(M, n, **f64)
        s["index"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["energy"], s["min_eig"], s["logdet"] = (torch.zeros(n, **f64) for _ in range(3))
        s["dup"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["dup_count"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind == "quadratic":
        eq, va, vb, coef, gamma = _quadratic(case, seed)
        s["system"] = nphc.System.quadratic(case["n"], eq, va, vb, coef)
        s["opts"] = nphc.options_default(gamma=gamma, precision=nphc.PREC_FP64)
        s["result"] = nphc.Result(s["system"])
    else:   # endgame
        gamma, J = _ring(case["N"], 0.0, seed)
        s["system"] = system = nphc.System(case["N"], J=J)
        s["opts"] = nphc.options_default(gamma=gamma)
        paths = np.random.default_rng(seed).choice(system.npaths, case["count"], replace=False)
        s["ep"] = nphc.DeviceEndpoints.empty(system.n, np.sort(paths))
        s["ws"] = torch.empty(system.workspace_size(case["count"]), dtype=torch.uint8, device="cuda")
        s["cycle"] = torch.zeros(case["count"], dtype=torch.int32, device="cuda")
        s["status"] = torch.zeros(case["count"], dtype=torch.int32, device="cuda")
    return s


def run(s):
    return globals()["_run_" + s["kind"]](s)


def _certified_counts(result):
    c = result.counts()
    return np.array([c[k] for k in ("paths", "real", "nonreal", "undecided", "singular", "duplicate")]
                    + c["index_hist"])


def _capacity(N):
    """Rows kept for the real stationary points of a ring (20 at N = 5, 4,774 at N = 11)."""
    return 1 << (N + 2)


def _turn(theta):
    """Angles modulo 2 pi, the branch cut away from 0 and pi."""
    lib = torch if isinstance(theta, torch.Tensor) else np
    return lib.remainder(theta + 1e-6, 2 * math.pi)


def _sps(result):
    p = result.stationary_points()
    p["theta"] = _turn(p["theta"])
    out = {}
    for k in ("theta", "energy", "index", "path", "log_abs_det"):
        out[k] = np.zeros((_capacity(result.system.N),) + p[k].shape[1:], p[k].dtype)
        out[k][:len(p[k])] = p[k]
    return out


def _solutions(result):
    e = result.endpoints()
    none = ~np.isin(e["cls"], CERTIFIED)
    e["cls"][none] = 0
    e["z"][none] = 0
    return dict(cls=e["cls"], z=e["z"])


def _run_solve(s):
    nphc.solve_into(s["system"], s["opts"], s["result"])
    out = _sps(s["result"]) if s["read"] == "sps" else _solutions(s["result"])
    out["counts"] = _certified_counts(s["result"])
    return out


def _run_batch(s):
    s["batch"].solve(s["opts"])
    results = [s["batch"].result(i) for i in range(len(s["systems"]))]
    sps = [_sps(r) for r in results]
    out = {k: np.concatenate([p[k].ravel() for p in sps]) for k in sps[0]}
    out["counts"] = np.concatenate([_certified_counts(r) for r in results])
    return out


def _run_chunk(s):
    system, opts, ep, ws = s["system"], s["opts"], s["ep"], s["ws"]
    nphc.track(system, opts, nphc.PREC_MIXED, ep, ws)
    st = ep.tensors["status"]
    todo = torch.nonzero((st == nphc.PATH_HANDOFF) | (st == nphc.PATH_HANDOFF_COND)).flatten().to(torch.int32)
    if todo.numel():
        count = torch.tensor([todo.numel()], dtype=torch.int32, device="cuda")
        nphc.track(system, opts, nphc.PREC_FP64, ep, ws, todo, count, resume=True)
    nphc.refine_certify(system, opts, ep)
    cls = ep.tensors["cls"]
    keep = (cls >= nphc.END_REAL) & (cls <= nphc.END_UNDECIDED)
    return dict(cls=cls * keep, z_re=torch.where(keep, ep.tensors["z_re"], 0.0),
                z_im=torch.where(keep, ep.tensors["z_im"], 0.0))


def _rows(v, N):
    """The rows of v in a buffer of the ring's capacity."""
    out = torch.zeros((_capacity(N),) + v.shape[1:], dtype=v.dtype, device=v.device)
    out[:len(v)] = v
    return out


def _run_gradient(s):
    s["value"].grad = None
    J = autograd.ring_couplings(s["N"], s["value"], s["g"], s["disorder"])
    energy, theta = autograd.stationary_points(J, s["gamma"])
    loss = energy.square().sum() + torch.sin(theta).sum()
    loss.backward()
    return dict(energy=_rows(energy.detach(), s["N"]), theta=_rows(_turn(theta.detach()), s["N"]),
                d_sigma=s["value"].grad)


def _run_adjoint(s):
    return nphc.xy_adjoint(s["system"], s["theta"], s["g_energy"], s["g_theta"])


def _run_certify(s):
    system, opts, ep = s["system"], s["opts"], s["ep"]
    t = ep.tensors
    t["z_re"].copy_(s["z_re"])
    t["z_im"].copy_(s["z_im"])
    t["status"].fill_(nphc.PATH_REACHED)
    nphc.refine_certify(system, opts, ep)
    nphc.dedup(system, opts, ep, s["ws"], s["dup"], s["dup_count"])
    nphc.classify(system, ep, s["theta"], s["index"], s["energy"], s["min_eig"], s["logdet"])
    return dict(z_re=t["z_re"], z_im=t["z_im"], cls=t["cls"], dup_count=s["dup_count"], theta=_turn(s["theta"]),
                index=s["index"], energy=s["energy"], min_eig=s["min_eig"], logdet=s["logdet"])


def _run_quadratic(s):
    nphc.solve_into(s["system"], s["opts"], s["result"])
    return _solutions(s["result"])


def _run_endgame(s):
    t = s["ep"].tensors
    nphc.endgame(s["system"], s["opts"], s["ep"], s["ws"], s["cycle"], s["status"])
    keep = s["status"] == nphc.EG_CONVERGED
    return dict(cycle=s["cycle"], status=s["status"], z_re=torch.where(keep, t["z_re"], 0.0),
                z_im=torch.where(keep, t["z_im"], 0.0))


# -------------------------------------------------------------------- work --
def _solve_flops(M):
    """One solve of the homotopy's linear system by its M x M Schur complement: the matrix's
    entries, an LU with one right-hand side, the change of variables."""
    return 8 * M ** 3 / 3 + 8 * M * M * 4 + 150 * M


SOLVES_PER_PATH = 250   # tracked with RK4 and Newton's corrector (N = 5 .. 12: 150 to 330)


def work(case):
    kind = case["kind"]
    if kind == "solve":
        P, M = 4 ** (case["N"] - 1), case["N"] - 1
        out = P * (32 * M + 4) if case["read"] == "solutions" else P * (8 * M + 36) / 150
        return dict(bytes=8 * case["N"] ** 2 + out, flops=P * SOLVES_PER_PATH * _solve_flops(M))
    if kind == "batch":
        sizes = range(case["lo"], case["hi"] + 1)
        each = case["count"] / len(sizes)
        return dict(bytes=sum(each * 4 ** (N - 1) * (8 * N + 28) / 150 for N in sizes),
                    flops=sum(each * 4 ** (N - 1) * SOLVES_PER_PATH * _solve_flops(N - 1) for N in sizes))
    if kind == "chunk":
        M = case["N"] - 1
        return dict(bytes=case["count"] * (8 + 4 + 32 * M),
                    flops=case["count"] * SOLVES_PER_PATH * _solve_flops(M))
    if kind == "gradient":
        P, M = 4 ** (case["N"] - 1), case["N"] - 1
        return dict(bytes=P * (8 * M + 8) / 50, flops=P * SOLVES_PER_PATH * _solve_flops(M))
    if kind == "adjoint":
        M = case["N"] - 1
        return dict(bytes=case["count"] * (16 * M + 8) + 8 * (M + 1) ** 2,
                    flops=case["count"] * (2 * M ** 3 / 3 + 12 * M * M + 80 * M))
    if kind == "certify":   # two Newton steps, the inverse's norm, and the real points' eigenvalues
        M = case["N"] - 1
        return dict(bytes=case["count"] * (32 * M * 2 + 8 * M + 36),
                    flops=case["count"] * (3 * _solve_flops(M) + 24 * M ** 3))
    if kind == "quadratic":
        n = case["n"]
        return dict(bytes=2 ** n * (16 * n + 4),
                    flops=2 ** n * SOLVES_PER_PATH * (8 * n ** 3 / 3 + n * case["terms"] * 30))
    M = case["N"] - 1   # endgame: tracking to its first radius, then two radii of 16 samples
    return dict(bytes=case["count"] * (16 * M * 2 + 16),
                flops=case["count"] * (100 + 2 * 16 * 4) * _solve_flops(M))


# ----------------------------------------------------------- exact values --
def exact(case, seed):
    kind = case["kind"]
    if kind == "adjoint":
        return _exact_adjoint(case, seed)
    if kind == "certify":
        return _exact_certify(case, seed)
    if kind == "solve" and case["N"] <= 6:
        gamma, J = _ring(case["N"], case["disorder"], seed, case["sigma"])
        z = _homotopy(*_ring_polynomials(J), gamma)
        if case["read"] == "solutions":
            return dict(cls=None, z=z, counts=None)
        th = _real_angles(z)
        H = _grad_hess(th, torch.as_tensor(J, device="cuda"))[1]
        return dict(theta=_rows(_turn(th), case["N"]), energy=_rows(_energy(th, J), case["N"]), index=None,
                    path=None, log_abs_det=_rows(torch.linalg.slogdet(H)[1], case["N"]), counts=None)
    if kind == "quadratic" and case["n"] <= 10:
        eq, va, vb, coef, gamma = _quadratic(case, seed)
        n = case["n"]
        Q, L, c = np.zeros((n, n, n), complex), np.zeros((n, n), complex), np.zeros(n, complex)
        for i, a, b, v in zip(eq, va, vb, coef):
            if a >= 0 and b >= 0:
                Q[i, a, b] += v
            elif a >= 0 or b >= 0:
                L[i, max(a, b)] += v
            else:
                c[i] += v
        return dict(cls=None, z=_homotopy(Q, L, c, gamma))
    if kind == "gradient" and case["N"] <= 6:
        return _exact_gradient(case, seed)
    return None


def _energy(th, J):
    J = torch.as_tensor(J, device=th.device)
    full = torch.cat([th, torch.zeros_like(th[:, :1])], 1)
    return 0.5 * (J * (1 - torch.cos(full[:, :, None] - full[:, None, :]))).sum((1, 2))


def _real_angles(z):
    """The angles of the real ones among the solutions (rows of zeros: none), in their order."""
    M = z.shape[1] // 2
    size = z.abs().amax(1)
    real = (size > 0) & (z.imag.abs().amax(1) < 1e-9 * (1 + size))
    return torch.atan2(z[real, M:].real, z[real, :M].real)


def _adjoint_inputs(case, J, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 2)
    theta = _angles(J, case["count"], seed).real.contiguous()
    f64 = dict(generator=gen, dtype=torch.float64, device="cuda")
    return theta, torch.randn(len(theta), **f64), torch.randn(theta.shape, **f64)


def _dJ(theta, g_energy, g_theta, J):
    """dL/dJ by the envelope theorem (V) and the implicit function theorem (theta)."""
    H = _grad_hess(theta, J)[1]
    lam = torch.linalg.solve(H, g_theta.unsqueeze(2)).squeeze(2)
    pad = torch.zeros_like(theta[:, :1])
    th, lam = torch.cat([theta, pad], 1), torch.cat([lam, pad], 1)
    d = th[:, :, None] - th[:, None, :]
    return (g_energy[:, None, None] * (1 - torch.cos(d))
            - (lam[:, :, None] - lam[:, None, :]) * torch.sin(d)).sum(0)


def _exact_adjoint(case, seed):
    _, J = _ring(case["N"], 0.1, seed)
    return _dJ(*_adjoint_inputs(case, J, seed), torch.as_tensor(J, device="cuda"))


def _exact_gradient(case, seed):
    rng = np.random.default_rng(seed)
    N = case["N"]
    g = inputs.draw_pair_normals(rng, N)
    gamma = inputs.draw_gamma(rng)
    sigma = float(rng.uniform(0.5, 3.0))
    J = _couplings(N, sigma, g, case["disorder"])
    th = _real_angles(_homotopy(*_ring_polynomials(J), gamma))
    Jt = torch.as_tensor(J, device="cuda")
    energy = _energy(th, J)
    dJ = _dJ(th, 2 * energy, torch.cos(th), Jt).cpu().numpy()
    i = np.arange(N)
    d = np.abs(i[:, None] - i[None, :])
    d = np.maximum(np.minimum(d, N - d), 1)
    return dict(energy=_rows(energy, N), theta=_rows(_turn(th), N), d_sigma=torch.tensor(float(0.5 * (dJ * -np.log(d) * J).sum()), dtype=torch.float64))


def _certify_points(case, J, seed):
    """[count, 2M] solutions (cos theta, sin theta) of the polynomial system."""
    th = _angles(J, case["count"], seed, complex_part=0.75)
    return torch.cat([torch.cos(th), torch.sin(th)], 1)


def _exact_certify(case, seed):
    _, J = _ring(case["N"], 0.1, seed)
    z = _certify_points(case, J, seed)
    n, M = z.shape[0], case["N"] - 1
    # the first of every group of copies keeps its class
    gen = torch.Generator(device="cuda").manual_seed(7)
    w = torch.randn(2 * M, generator=gen, device="cuda", dtype=torch.complex128)
    key = torch.round(torch.view_as_real(z @ w) * 1e6).to(torch.int64).cpu().numpy()
    first = np.unique(key, axis=0, return_index=True)[1]
    real = z.imag.abs().amax(1) < 1e-9
    kept = torch.zeros(n, dtype=torch.bool, device="cuda")
    kept[torch.as_tensor(first, device="cuda")] = True
    kept &= real
    th = torch.atan2(z[kept, M:].real, z[kept, :M].real)
    ev = torch.linalg.eigvalsh(_grad_hess(th, torch.as_tensor(J, device="cuda"))[1])
    out = dict(z_re=z.real.T, z_im=z.imag.T, cls=None, dup_count=None, index=None)
    for name, v in (("energy", _energy(th, J)), ("min_eig", ev.abs().amin(1)),
                    ("logdet", ev.abs().log().sum(1)), ("theta", _turn(th))):
        full = torch.full((n,) + v.shape[1:], 1e-6 if name == "theta" else 0.0, dtype=torch.float64, device="cuda")
        full[kept] = v
        out[name] = full.movedim(0, -1)
    return out


def _ring_polynomials(J):
    """The ring's equations as (Q, L, c): P_i(z) = z Q_i z + L_i z + c_i, z = (x, y)."""
    N = len(J)
    M = N - 1
    Q, L, c = np.zeros((2 * M, 2 * M, 2 * M), complex), np.zeros((2 * M, 2 * M), complex), np.zeros(2 * M, complex)
    for k in range(M):
        for j in range(M):
            if j != k:
                Q[k, M + k, j] += J[k, j]
                Q[k, k, M + j] -= J[k, j]
        L[k, M + k] += J[k, M]
        Q[M + k, k, k] = Q[M + k, M + k, M + k] = 1
        c[M + k] = -1
    return Q, L, c


def _homotopy(Q, L, c, gamma):
    """The nonsingular solutions at t = 1 of gamma (1 - t)(z^2 - 1) + t P(z), one row per
    start point (bit i of the index: z_i = -1), zeros where a path has none: RK4 and Newton
    on all paths at once, each with its own step."""
    n = len(c)
    Q, L, c = (torch.as_tensor(v, device="cuda") for v in (Q + Q.transpose(0, 2, 1), L, c))

    def parts(z):
        Qz = torch.einsum("iab,pb->pia", Q, z)
        return 0.5 * (Qz * z[:, None, :]).sum(2) + z @ L.T + c, Qz + L

    def solve(z, t, rhs_t):
        P, DP = parts(z)
        a = (gamma * (1 - t))[:, None]
        H = torch.diag_embed(2 * a * z) + t[:, None, None] * DP
        r = gamma * (z * z - 1) - P if rhs_t else -(a * (z * z - 1) + t[:, None] * P)
        return torch.linalg.solve_ex(H, r.unsqueeze(2))[0].squeeze(2)

    index = torch.arange(2 ** n, device="cuda")
    z = (1 - 2.0 * ((index[:, None] >> torch.arange(n, device="cuda")) & 1)).to(torch.complex128)
    t = torch.zeros(len(z), dtype=torch.float64, device="cuda")
    h = torch.full_like(t, 0.01)
    run = torch.zeros_like(index)
    end = torch.full_like(z, math.nan)
    for _ in range(2500):
        if not len(z):
            break
        t1 = torch.clamp(t + h, max=1.0)
        d = (t1 - t)[:, None]
        tm = 0.5 * (t + t1)
        k1 = solve(z, t, True)
        k2 = solve(z + 0.5 * d * k1, tm, True)
        k3 = solve(z + 0.5 * d * k2, tm, True)
        w = z + d / 6 * (k1 + 2 * k2 + 2 * k3 + solve(z + d * k3, t1, True))
        first = step = solve(w, t1, False)
        for _ in range(2):
            w = w + step
            step = solve(w, t1, False)
        w = w + step
        norm = 1 + w.norm(dim=1)
        good = (first.norm(dim=1) < 1e-2 * norm) & (step.norm(dim=1) < 1e-10 * norm)
        z = torch.where(good[:, None], w, z)
        t = torch.where(good, t1, t)
        run = torch.where(good, run + 1, 0)
        grow = run >= 3
        run = torch.where(grow, 0, run)
        h = torch.where(good, torch.where(grow, 2 * h, h).clamp(max=0.05), 0.5 * h)
        far = z.abs().amax(1) > 1e8
        done = t >= 1
        end[index[done & ~far]] = z[done & ~far]
        on = ~done & ~far & (h > 1e-15)
        index, z, t, h, run = index[on], z[on], t[on], h[on], run[on]
    one = torch.ones(len(end), dtype=torch.float64, device="cuda")
    for _ in range(3):
        end = end + solve(end, one, False)
    cond = torch.linalg.matrix_norm(parts(end)[1]) * torch.linalg.matrix_norm(torch.linalg.inv_ex(parts(end)[1])[0])
    return torch.where((cond < 1e11 * end.abs().amax(1).clamp(min=1) ** 2)[:, None], end, 0)
