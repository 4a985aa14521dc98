"""Timing cases of the library: what a user's program has it do, over the real
range of sizes, precisions, routes and options.

A case is a dict of plain values.  `kind` selects the entry point:

* "solve":  bec_gmres_solve on a constant-coefficient heat problem (sine-transform
            route), 1D, 2D or 3D, finite differences or Q1, BDF1 or BDF2;
* "apply":  bec_apply_Pinv alone, for programs with a Krylov method of their own;
* "mg":     bec_gmres_solve with a variable coefficient a = exp(Gaussian field)
            (multigrid route);
* "wind":   bec_gmres_solve of convection-diffusion (Example 3 of Sec. 5) on the
            ILU-smoothed multigrid;
* "batch":  bec_batch_solve of uneven instances;
* "grad":   bec_learned_loss_grad, the training step's loss and weight gradient.

nx + 1 and N are powers of two everywhere (the library takes no others).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2002_01108_gb300 import Batch, Problem


def _solve(name, dim, m, N, eps, precision="fp64", **kw):
    case = {"name": name, "kind": "solve", "dim": dim, "m": m, "N": N, "eps": eps, "a": 1.0,
            "precision": precision, "space": "fd", "scheme": "bdf1", "restart": 30,
            "rtol": 1e-8, "flexible": True, "left": False}
    case.update(kw)
    return case


def listed():
    return [
        # the smallest configuration: a call made of launches and latencies
        _solve("solve1d_63_N64_fp64", 1, 63, 64, 0.5 / 8.0, rtol=1e-10, flexible=False),
        # an ordinary small solve, Q1 elements and left GMRES as in the paper's table
        _solve("solve2d_q1_127_N64_fp64", 2, 127, 64, 0.5 / 64, a=1e-5, space="q1", restart=50,
               rtol=1e-7, flexible=False, left=True),
        # the benchmark workload, plain FP64 and mixed precision
        _solve("solve2d_255_N256_fp64", 2, 255, 256, 1.0 / 16),
        _solve("solve2d_255_N256_fp32", 2, 255, 256, 1.0 / 16, precision="fp32"),
        # the largest: 133.7M unknowns in mixed precision
        _solve("solve2d_511_N512_fp32", 2, 511, 512, math.sqrt(1.0 / 512), precision="fp32",
               restart=20),
        # a cube
        _solve("solve3d_31_N128_fp64", 3, 31, 128, math.sqrt(1.0 / 128)),
        # the preconditioner alone, both precisions
        {"name": "apply2d_255_N256_fp64", "kind": "apply", "dim": 2, "m": 255, "N": 256,
         "eps": 1.0 / 16, "a": 1.0, "precision": "fp64", "space": "fd", "scheme": "bdf1"},
        {"name": "apply2d_255_N256_fp32", "kind": "apply", "dim": 2, "m": 255, "N": 256,
         "eps": 1.0 / 16, "a": 1.0, "precision": "fp32", "space": "fd", "scheme": "bdf1"},
        # variable coefficient: the fastest multigrid form, and FP64 as the plain form
        {"name": "mg2d_255_N256_fp32", "kind": "mg", "m": 255, "N": 256, "eps": 1.0 / 32,
         "precision": "fp32", "pre": 3, "post": 2, "rtol": 1e-8},
        {"name": "mg2d_127_N64_fp64", "kind": "mg", "m": 127, "N": 64, "eps": 1.0 / 16,
         "precision": "fp64", "pre": 1, "post": 1, "rtol": 1e-8},
        # convection-diffusion with the ILU smoother
        {"name": "wind2d_127_N128_fp32", "kind": "wind", "m": 127, "N": 128, "eps": 0.5 / 128,
         "precision": "fp32", "rtol": 1e-8},
        # many uneven instances at once, as a serving program has them
        {"name": "batch12_fp32", "kind": "batch", "count": 12, "pick": 4, "mode": "graphs",
         "nstreams": 8},
    ]


def _log_eps(rng, N):
    """eps ~ logU[1e-4, sqrt(tau)]."""
    lo, hi = math.log(1e-4), math.log(math.sqrt(1.0 / N))
    return math.exp(rng.uniform(lo, hi))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "apply", "apply", "mg", "batch", "wind", "grad"])
    if kind in ("solve", "apply"):
        dim = rng.choice([1, 2, 2, 2, 3])
        logn = {1: rng.randint(4, 10), 2: rng.randint(4, 9), 3: rng.randint(3, 6)}[dim]
        # at most 2^25 unknowns, a quarter of the largest listed solve
        logt = rng.randint(3, max(3, min(10, 25 - dim * logn)))
        N = 1 << logt
        case = {"kind": kind, "dim": dim, "m": (1 << logn) - 1, "N": N, "eps": _log_eps(rng, N),
                "a": math.exp(rng.uniform(math.log(1e-2), 0.0)),
                "precision": rng.choice(["fp64", "fp64", "fp32"]),
                "space": rng.choice(["fd", "fd", "q1"]) if dim < 3 else "fd",
                "scheme": rng.choice(["bdf1", "bdf1", "bdf2"]) if dim < 3 else "bdf1"}
        if kind == "solve":
            left = case["precision"] == "fp64" and rng.random() < 0.25
            case.update(restart=20, rtol=rng.choice([1e-8, 1e-8, 1e-10]), left=left,
                        flexible=case["precision"] == "fp32" or (not left and rng.random() < 0.5))
        return case
    if kind == "mg":
        logn = rng.randint(5, 8)
        logt = rng.randint(4, 22 - 2 * logn if logn > 6 else 9)
        N = 1 << logt
        return {"kind": "mg", "m": (1 << logn) - 1, "N": N, "eps": _log_eps(rng, N),
                "precision": rng.choice(["fp32", "fp64"]), "pre": rng.randint(1, 3),
                "post": rng.randint(1, 2), "rtol": 1e-8}
    if kind == "wind":
        logn = rng.randint(5, 7)
        N = 1 << rng.randint(4, 7)
        return {"kind": "wind", "m": (1 << logn) - 1, "N": N, "eps": _log_eps(rng, N),
                "precision": rng.choice(["fp32", "fp32", "fp64"]), "rtol": 1e-8}
    if kind == "grad":
        return {"kind": "grad", "m": rng.choice([31, 63, 127]), "N": 1 << rng.randint(4, 6),
                "B": rng.randint(1, 32)}
    return {"kind": "batch", "count": rng.randint(2, 10), "pick": rng.randrange(1 << 30),
            "mode": rng.choice(["graphs", "streams", "persistent"]), "nstreams": rng.choice([1, 4, 8])}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(shape, g):
    return torch.rand(shape, dtype=torch.float64, device="cuda", generator=g).mul_(2.0).sub_(1.0)


def _sines(m, count):
    x = torch.arange(1, m + 1, dtype=torch.float64, device="cuda") / (m + 1)
    j = torch.arange(1, count + 1, dtype=torch.float64, device="cuda")
    return torch.sin(math.pi * x[:, None] * j[None, :])


def _u0(dim, m, g):
    """A random sine series of 8 terms a dimension."""
    c = _uniform((8,) * dim, g)
    s = _sines(m, 8)
    for d in range(dim):
        c = torch.movedim(torch.tensordot(s, c, dims=([1], [d])), 0, d)
    return c.contiguous()


def _field(m, seed, ell=0.1):
    """Log coefficient: a Gaussian random field with squared-exponential
    covariance on all (m + 2)^2 nodes."""
    rng = np.random.default_rng(seed)
    x = np.arange(m + 2) / (m + 1)
    d, q = np.linalg.eigh(np.exp(-np.subtract.outer(x, x) ** 2 / (2.0 * ell * ell)))
    r = q * np.sqrt(np.maximum(d, 0.0))
    return r @ rng.standard_normal((m + 2, m + 2)) @ r.T


def _wind_data(m, N):
    """Example 3: the circulating wind, and the hot wall's boundary values."""
    s = -1.0 + 2.0 * np.arange(m + 2) / (m + 1)
    X, Y = np.meshgrid(s, s)
    wind = np.stack([2.0 * Y * (1.0 - X * X), -2.0 * X * (1.0 - Y * Y)])
    phi = torch.zeros((m + 2, m + 2), dtype=torch.float64, device="cuda")
    phi[:, m + 1] = 1.0
    t = torch.arange(1, N + 1, dtype=torch.float64, device="cuda") / N
    return wind, (1.0 - torch.exp(-10.0 * t))[:, None, None] * phi


def _instances(case):
    """The uneven instances of a batch (sides, steps and eps as in the batch
    workload), at most 2^24 unknowns in all."""
    rng = np.random.default_rng(case["pick"])
    out, total = [], 0
    for _ in range(case["count"]):
        m, N = int(rng.choice((63, 127, 255))), int(rng.choice((32, 64, 128, 256, 512)))
        while m * m * N + total > (1 << 24) and (m > 63 or N > 32):
            m, N = (m // 2, N) if m > 63 else (m, N // 2)
        total += m * m * N
        out.append({"dim": 2, "nx": m, "N": N, "precision": "fp32", "max_restart": 10,
                    "eps": math.exp(rng.uniform(math.log(1e-4), math.log(math.sqrt(1.0 / N))))})
    return out


# ------------------------------------------------------------------ prepare
def _heat_problem(case):
    p = Problem(case["dim"], case["m"], case["N"], a=case["a"], precision=case["precision"],
                max_restart=case.get("restart", 2), flexible=case.get("flexible", False),
                space=case["space"], scheme=case["scheme"])
    p.set_eps(case["eps"])
    p.autotune()
    return p


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    if kind == "apply":
        p = _heat_problem(case)
        return {"case": case, "p": p, "y": _uniform(p.shape, g), "z": p._new()}
    if kind == "solve":
        p = _heat_problem(case)
        u0 = _u0(case["dim"], case["m"], g)
        f = p.build_rhs(u0, _uniform(p.shape, g))
        return {"case": case, "p": p, "f": f, "u": torch.empty_like(f),
                "kw": dict(restart=case["restart"], rtol=case["rtol"], maxit=300,
                           flexible=case["flexible"], left_pc=case["left"])}
    if kind in ("mg", "wind"):
        m, N = case["m"], case["N"]
        if kind == "mg":
            p = Problem(2, m, N, route="mg", a_nodes=np.exp(_field(m, seed)),
                        precision=case["precision"], flexible=True, max_restart=30,
                        mg_pre=case["pre"], mg_post=case["post"])
            p.set_eps(case["eps"])
            u0 = _u0(2, m, g)
            f = p.build_rhs(u0, _uniform(p.shape, g))
        else:
            wind, walls = _wind_data(m, N)
            p = Problem(2, m, N, a=1.0 / 200.0, route="mg", wind=wind, side=2.0,
                        mg_smoother="ilu", precision=case["precision"], flexible=True,
                        max_restart=30)
            p.set_eps(case["eps"])
            f = p.build_rhs_dirichlet(_u0(2, m, g), _uniform(p.shape, g), walls)
        return {"case": case, "p": p, "f": f, "u": torch.empty_like(f),
                "kw": dict(restart=30, rtol=case["rtol"], maxit=300, flexible=True)}
    if kind == "grad":
        m, N, B = case["m"], case["N"], case["B"]
        p = Problem(2, m, N, route="learned", precision="fp32", a_nodes=np.exp(_field(m, seed)),
                    flexible=True, max_restart=2)
        p.set_eps(1.0 / 16)
        mc = (m - 1) // 2
        return {"case": case, "p": p,
                "lam": [int(k) for k in np.random.default_rng(seed).integers(0, N // 2 + 1, B)],
                "r": torch.view_as_complex(_uniform((B, m, m, 2), g)),
                "e": torch.view_as_complex(_uniform((B, mc, mc, 2), g))}
    specs = _instances(case)
    b = Batch(specs, nstreams=case["nstreams"], mode=case["mode"])
    fs = []
    for i, s in enumerate(specs):
        shape = (s["N"], s["nx"], s["nx"])
        u0 = _u0(2, s["nx"], g)
        src = _uniform(shape, g)
        torch.cuda.synchronize()                    # the instance has a stream of its own
        fs.append(b.build_rhs(i, u0, src, torch.empty(shape, dtype=torch.float64, device="cuda")))
        torch.cuda.synchronize()
    return {"case": case, "b": b, "fs": fs, "us": [torch.empty_like(f) for f in fs]}


# ------------------------------------------------------------------ run
def run(state):
    kind = state["case"]["kind"]
    if kind == "apply":
        return state["p"].apply_Pinv(state["y"], state["z"])
    if kind == "grad":
        loss, grad = state["p"].learned_loss_grad(state["lam"], state["r"], state["e"])
        return {"loss": np.array([loss], dtype=np.float32), "grad": grad}
    if kind == "batch":
        infos = state["b"].solve(state["fs"], state["us"], restart=10, rtol=1e-8)
        return {"u": state["us"], "converged": [i["converged"] for i in infos]}
    u, info = state["p"].gmres_solve(state["f"], state["u"], **state["kw"])
    return {"u": u, "iters": info["iters"], "converged": info["converged"]}


# ------------------------------------------------------------------ work
def work(case):
    """Bytes: the right-hand side read and the solution written.  Flops: one
    P_eps^{-1} (a transform of n points as 2.5 n log2 n) and one product with L."""
    kind = case["kind"]
    if kind == "batch":
        w = [work({"kind": "solve", "dim": 2, "m": s["nx"], "N": s["N"]}) for s in _instances(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "grad":
        m, B = case["m"], case["B"]
        mc = (m - 1) // 2
        # 3 x 3 convolutions over the network's levels, forward and twice that backward
        pix = 2 * B * mc * mc
        return {"bytes": 16.0 * B * (m * m + mc * mc), "flops": 3.0 * pix * 2 * 9 * 32 * 32 * 2.5}
    dim, m, N = case.get("dim", 2), case["m"], case["N"]
    U = float(m ** dim * N)
    fft_t = 2 * 2.5 * math.log2(N) + 8
    if kind in ("mg", "wind"):
        # per frequency (half of N) and point: two smoothings and a residual, all levels
        flops = U * (fft_t + 0.5 * (2 * 98 + 84) * 4 / 3 + 9)
    else:
        flops = U * (2 * dim * 2.5 * math.log2(2 * (m + 1)) + fft_t)
        if kind == "solve":
            flops += U * (2 * dim + 3)
    return {"bytes": 16.0 * U, "flops": flops}


# ------------------------------------------------------------------ exact
def _dst(v, m, axes):
    """Orthonormal sine transform along the given axes."""
    k = torch.arange(1, m + 1, dtype=torch.float64, device="cuda")
    # the angle is reduced modulo 2 pi in whole numbers
    s = torch.sin(math.pi / (m + 1) * torch.remainder(k[:, None] * k[None, :], 2 * (m + 1)))
    s *= math.sqrt(2.0 / (m + 1))
    for ax in axes:
        v = torch.movedim(torch.matmul(torch.movedim(v, ax, -1), s), -1, ax)
    return v


def _eigs(case, h):
    """Mass and stiffness eigenvalues on the sine basis, shaped like a slice."""
    dim, m = case["dim"], case["m"]
    k = torch.arange(1, m + 1, dtype=torch.float64, device="cuda")
    s2 = torch.sin(k * (math.pi * h / 2)) ** 2
    if case["space"] == "q1":
        kk, mm = case["a"] * 4.0 / h * s2, h / 3.0 * (2.0 + torch.cos(k * (math.pi * h)))
        if dim == 1:
            return mm, kk
        return mm[:, None] * mm, mm[:, None] * kk + kk[:, None] * mm
    kk = case["a"] * 4.0 / h ** 2 * s2
    tot = kk
    for _ in range(dim - 1):
        tot = tot[..., None] + kk
    return torch.ones_like(tot), tot


def _march(fh, mm, kk, tau, bdf2):
    """L^{-1} f, mode by mode, one time step after the other, in place."""
    r0 = 1.5 if bdf2 else 1.0
    d = r0 * mm + tau * kk
    for n in range(fh.shape[0]):
        if n > 0:
            fh[n] += (2.0 if bdf2 else 1.0) * mm * fh[n - 1]
        if bdf2 and n > 1:
            fh[n] -= 0.5 * mm * fh[n - 2]
        fh[n] /= d
    return fh


def _exact_heat(case, f):
    dim, m, N = case["dim"], case["m"], case["N"]
    axes = range(1, dim + 1)
    mm, kk = _eigs(case, 1.0 / (m + 1))
    return _dst(_march(_dst(f, m, axes).contiguous(), mm, kk, 1.0 / N, case["scheme"] == "bdf2"),
                m, axes)


def _exact_apply(case, y):
    dim, m, N, eps = case["dim"], case["m"], case["N"], case["eps"]
    axes = range(1, dim + 1)
    mm, kk = _eigs(case, 1.0 / (m + 1))
    j = torch.arange(N, dtype=torch.float64, device="cuda")
    d = torch.pow(torch.tensor(eps, dtype=torch.float64, device="cuda"), j / N)
    e1 = eps ** (1.0 / N)
    th = torch.polar(torch.full_like(j, e1), -2.0 * math.pi * j / N)
    lam = 1.5 - 2.0 * th + 0.5 * th * th if case["scheme"] == "bdf2" else 1.0 - th
    shape = (N,) + (1,) * dim
    yh = _dst(y, m, axes)
    c = torch.fft.fft(yh * d.reshape(shape), dim=0)
    for k in range(N):
        c[k] /= lam[k] * mm + (1.0 / N) * kk
    return _dst(torch.fft.ifft(c, dim=0).real / d.reshape(shape), m, axes)


def _rhs(case, u0, src, mm=None):
    """tau f^n, plus M u^0 terms in the first rows."""
    N, dim, m = case["N"], case["dim"], case["m"]
    f = src / N
    mu0 = u0
    if case["space"] == "q1":
        axes = range(dim)
        mu0 = _dst(mm * _dst(u0, m, axes), m, axes)
    if case["scheme"] == "bdf2":
        f[0] += 1.5 * mu0
        f[1] -= 0.5 * mu0
    else:
        f[0] += mu0
    return f


def _exact_mg(case, seed, g):
    """Sequential time stepping, each step by conjugate gradients to 1e-14."""
    m, N = case["m"], case["N"]
    tau, h = 1.0 / N, 1.0 / (m + 1)
    a = torch.from_numpy(np.exp(_field(m, seed))).cuda()
    u0 = _u0(2, m, g)
    src = _uniform((N, m, m), g)
    c = tau / (h * h)
    ax = 0.5 * c * (a[1:-1, 1:] + a[1:-1, :-1])      # faces between x neighbours
    ay = 0.5 * c * (a[1:, 1:-1] + a[:-1, 1:-1])
    diag = 1.0 + ax[:, 1:] + ax[:, :-1] + ay[1:] + ay[:-1]

    def op(v):
        w = diag * v
        w[:, 1:] -= ax[:, 1:-1] * v[:, :-1]
        w[:, :-1] -= ax[:, 1:-1] * v[:, 1:]
        w[1:] -= ay[1:-1] * v[:-1]
        w[:-1] -= ay[1:-1] * v[1:]
        return w

    out, prev = torch.empty((N, m, m), dtype=torch.float64, device="cuda"), u0
    for n in range(N):
        b = tau * src[n] + prev
        x = prev.clone()
        r = b - op(x)
        z = r / diag
        p, rz, stop = z, (r * z).sum(), 1e-28 * (b * b).sum()
        for it in range(1, 4000):
            q = op(p)
            al = rz / (p * q).sum()
            x = x + al * p
            r = r - al * q
            if it % 50 == 0 and bool((r * r).sum() <= stop):
                break
            z = r / diag
            rz1 = (r * z).sum()
            p, rz = z + (rz1 / rz) * p, rz1
        out[n] = prev = x
    return out


def exact(case, seed):
    kind, g = case["kind"], _gen(seed)
    shape = (case.get("N"),) + (case.get("m"),) * case.get("dim", 2)
    if kind == "apply":
        return _exact_apply(case, _uniform(shape, g))
    if kind == "solve":
        u0 = _u0(case["dim"], case["m"], g)
        mm, _ = _eigs(case, 1.0 / (case["m"] + 1))
        return {"u": _exact_heat(case, _rhs(case, u0, _uniform(shape, g), mm)),
                "iters": None, "converged": None}
    if kind == "mg" and case["m"] * case["N"] <= 127 * 64:
        return {"u": _exact_mg(case, seed, g), "iters": None, "converged": None}
    if kind == "batch":
        us = []
        for s in _instances(case):
            one = {"dim": 2, "m": s["nx"], "N": s["N"], "a": 1.0, "space": "fd", "scheme": "bdf1"}
            u0 = _u0(2, s["nx"], g)
            us.append(_exact_heat(one, _rhs(one, u0, _uniform((s["N"], s["nx"], s["nx"]), g))))
        return {"u": us, "converged": None}
    return None
