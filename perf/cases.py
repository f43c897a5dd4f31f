"""The performance cases: what a user of the solver has it do, at the sizes it is used at.

A solve case is a fixed number of flexible GMRES steps of the production
solve (at least one whole restart cycle, with its solution update and true
residual) through ``Solver.solve``: every kernel of a converged solve in the
proportions of one, at a length at which two correct codes still agree to
rounding (after a thousand steps of restarted GMRES the last bits of the
iterates are noise).  The other cases are the calls a full-waveform inversion
makes beside the solves: operator, preconditioner, misfit and gradient.

Results of the mixed mode are kept in complex64, as a program that stores
wavefields does.  Its cycles are FP32: the preconditioner's output holds FP32
values (the conversion loses nothing), and the iterate carries their rounding
(the same solve with b scaled by 1 + 2^-30 differs by 5e-8 to 2.5e-7 after the
scaling is divided out, where a plain FP64 solve differs by 1e-15).  Results of
the FP64 mode, the operator and the gradient stay in FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2411_15897_gb300 as bah
import workloads as W
from paper_2411_15897_gb300.misfit import receiver_indices

# what a solve case means where it says nothing else: the library's defaults
# (V(1,2), FGMRES(20), one source, FP64 basis) with the benchmark's mixed mode
DEFAULTS = dict(medium="layered", n3=0, levels=0, cycle="V", nu_pre=1, nu_post=2, alpha=-1.0, restart=20, steps=20,
                precision="mixed", basis="fp64", sources=1, block=False, adjoint=False, host=False)


def listed():
    return [
        # the smallest call: a 64x64 grid, where every launch and every wait counts
        # (quick looks, tests, the first grids of a frequency sweep)
        dict(name="solve_64", kind="solve", medium="homogeneous", n1=64, n2=64),
        # the paper's linear medium (Table 4): an elongated grid with h1 != h2, no power
        # of two, W(1,2) and FGMRES(5); the adjoint solve of an inversion
        dict(name="solve_adjoint_400x128_w", kind="solve", medium="linear", n1=400, n2=128, levels=4, cycle="W",
             restart=5, steps=15, adjoint=True),
        # the benchmark: 512x512 layered medium, V(1,3), FGMRES(10), mixed precision,
        # vectors on the device
        dict(name="solve_512", kind="solve", n1=512, n2=512, nu_post=3, alpha=0.8, restart=10),
        # the same solve in plain FP64, the mode to check a mixed result with, through pinned
        # host buffers
        dict(name="solve_512_fp64_host", kind="solve", n1=512, n2=512, nu_post=3, alpha=0.8, restart=10,
             precision="fp64", host=True),
        # the smooth random medium at 1024x1024, seven levels, FGMRES(20): one large
        # single-source solve
        dict(name="solve_1024", kind="solve", medium="grf", n1=1024, n2=1024, nu_post=3, alpha=0.8),
        # a shot gather: 32 sources of the 1024x512 layered medium in one lockstep batch,
        # the largest call
        dict(name="solve_sources_1024x512x32", kind="solve", n1=1024, n2=512, sources=32),
        # eight sources in one Krylov space (block FGMRES)
        dict(name="solve_block_256x128x8", kind="solve", n1=256, n2=128, sources=8, block=True),
        # the 3-D workload: 128^3 random medium, W(2,2), mixed intergrid, five levels
        dict(name="solve_3d_128", kind="solve", medium="grf", n1=128, n2=128, n3=128, levels=5, cycle="W", nu_pre=2,
             nu_post=2, alpha=0.4),
        # a ragged 3-D grid of a smaller survey, three levels, coarsest 12 x 10 x 7
        dict(name="solve_3d_48x40x28", kind="solve", medium="grf", n1=48, n2=40, n3=28, levels=3, cycle="W", nu_pre=2,
             nu_post=2),
        # the preconditioner by itself, as an outer method of the user's own calls it, on a
        # grid that halves only three times (coarsest 45 x 25, a dense inverse of 1125 rows)
        dict(name="precond_360x200x4", kind="precond", n1=360, n2=200, sources=4),
        # H x and H^H x of a few vectors at 1024x1024: residuals and products of the user's own
        dict(name="operator_1024x4", kind="operator", medium="grf", n1=1024, n2=1024, sources=4),
        # misfit, adjoint sources and gradient of the shot gather
        dict(name="gradient_1024x512x32", kind="gradient", n1=1024, n2=512, sources=32),
    ]


def _size(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _axis(rng, size, levels):
    """A cell count near ``size`` that halves ``levels - 1`` times, odd or even below that."""
    f = 1 << (levels - 1)
    return max(4, round(size / f)) * f


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "block", "solve3", "precond", "operator", "gradient"])
    side = _size(rng, 64, 1024)
    ratio = rng.uniform(0.4, 1.0)
    # as many levels as leave 4 to 16 points on the coarsest grid's short side
    levels = max(2, int(math.log2(side * ratio / rng.uniform(5, 11))) + 1)
    n1, n2 = _axis(rng, side, levels), _axis(rng, side * ratio, levels)
    medium = rng.choice(["layered", "grf", "linear"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    c = dict(kind="solve", medium=medium, n1=n1, n2=n2, levels=levels)
    if kind == "solve":
        m = rng.choice([5, 10, 20])
        c.update(nu_pre=rng.choice([1, 1, 2]), nu_post=rng.choice([2, 3]), alpha=rng.choice([0.6, 0.8, 1.0]), restart=m,
                 steps=max(m, 10), precision=precision, cycle=rng.choice(["V", "V", "W"]),
                 basis=rng.choice(["fp64", "fp64", "df"]), adjoint=rng.random() < 0.3, host=precision == "fp64" and rng.random() < 0.5)
    elif kind == "batch":
        c.update(n1=_axis(rng, side / 2, levels - 1), n2=_axis(rng, side * ratio / 2, levels - 1),
                 levels=max(2, levels - 1), medium="layered", sources=rng.randint(2, 32), precision=precision,
                 restart=rng.choice([10, 20]), adjoint=rng.random() < 0.3)
    elif kind == "block":
        f = rng.choice([3, 4])
        c.update(n1=_axis(rng, _size(rng, 64, 256), f), n2=_axis(rng, _size(rng, 48, 128), f), levels=f, medium="layered",
                 sources=rng.randint(2, 12), block=True, steps=10)
    elif kind == "solve3":
        levels = rng.choice([2, 3, 4])
        f = 1 << (levels - 1)
        dims = [max(4, min(8, round(_size(rng, 24, 96) / f))) * f for _ in range(3)]
        c.update(n1=dims[0], n2=dims[1], n3=dims[2], levels=levels, medium="grf", cycle=rng.choice(["V", "W"]), nu_pre=2,
                 nu_post=2, precision=precision)
    elif kind == "precond":
        c.update(kind="precond", sources=rng.randint(1, 6), precision=precision)
    elif kind == "operator":
        c.update(kind="operator", sources=rng.randint(1, 8))
    else:
        c.update(kind="gradient", medium="layered", sources=rng.randint(1, 32))
    return c


def _problem(c, seed):
    n1, n2, n3 = c["n1"], c["n2"], c["n3"]
    abc = max(2, min(20, n2 // 8))
    if n3:
        return W.grf_medium((n1, n2, n3), max(4.0, n1 / 8.0), 2 * seed + 3, 2 * seed + 4, 8.0, max(2, min(10, n3 // 8)))
    if c["medium"] == "homogeneous":
        return W.homogeneous(n1, n2, 1.0, 2.0 * (1.0 + 0.01 * (seed % 97)), 0.25, 10.0, abc)
    if c["medium"] == "linear":
        return W.linear_medium(n1, n2, omega=1.75 * math.pi * n1 / 200.0, lam_factor=1.0 + 0.01 * (seed % 97), abc=abc)
    if c["medium"] == "grf":
        return W.grf_medium((n1, n2), n1 / 32.0, 2 * seed + 3, 2 * seed + 4, 10.0, abc)
    return W.layered(n1, n2, 6, seed + 2, abc=abc)


def _full(case):
    return {**DEFAULTS, **case}


def _solver(c, prob):
    opts = dict(precision=bah.BAH_MIXED if c["precision"] == "mixed" else bah.BAH_FP64, levels=c["levels"],
                cycle=bah.BAH_CYCLE_W if c["cycle"] == "W" else bah.BAH_CYCLE_V, nu_pre=c["nu_pre"],
                nu_post=c["nu_post"], shift_alpha=c["alpha"], restart=c["restart"], maxit=c["steps"],
                krylov_arith=bah.BAH_KRYLOV_DF if c["basis"] == "df" else bah.BAH_KRYLOV_FP64)
    if c["n3"]:
        opts.update(intergrid=bah.BAH_INTERGRID_MIXED, jacobi_w=(0.8, 0.8, 0.2))
    if c["kind"] == "solve":
        opts.update(rhs_block=c["sources"], block_krylov=int(c["block"]))
    return bah.Solver.from_problem(prob, **opts)


def _shots(c, prob, seed):
    """One vertical point force per source, on a row below the absorbing layer, spread along x_1."""
    rng = np.random.default_rng(seed)
    n, k = prob.n, c["sources"]
    shape = W.padded_shape(n)
    b = np.zeros((k,) + shape, dtype=np.complex128)
    row = max(1, prob.meta.get("abc", 2))
    for s in range(k):
        i = int((s + rng.uniform(0.2, 0.8)) * n[0] / k)
        idx = (row, i) if len(n) == 2 else (row, int(rng.uniform(0.3, 0.7) * n[1]), i)
        b[(s, len(n) - 1) + idx] = -1.0 / float(np.prod(prob.h))
    return torch.from_numpy(b if k > 1 else b[0])


def _fields(c, prob, seed, count):
    """Smooth-amplitude random vectors (boundary-normal entries zero), made on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn((count,) + W.padded_shape(prob.n), dtype=torch.complex128, device="cuda", generator=g)
    v[:, 0, :, 0] = 0
    v[:, 1, 0, :] = 0
    return v


def prepare(case, seed):
    c = _full(case)
    prob = _problem(c, seed)
    st = dict(c=c, solver=_solver(c, prob))
    if c["kind"] == "solve":
        b = _shots(c, prob, seed)
        st["b"] = b.pin_memory() if c["host"] else b.cuda()
        st["x"] = torch.zeros_like(b, pin_memory=True) if c["host"] else None
    elif c["kind"] == "gradient":
        k = c["sources"]
        st["x"], st["y"] = _fields(c, prob, seed, k), _fields(c, prob, seed + 1000003, k)
        rec = receiver_indices(prob.n, max(1, prob.meta["abc"]))
        st["rec"] = torch.from_numpy(rec).cuda()
        g = torch.Generator(device="cuda").manual_seed(seed + 7)
        st["d"] = torch.randn((k, len(rec)), dtype=torch.complex128, device="cuda", generator=g)
    else:
        st["x"] = _fields(c, prob, seed, c["sources"])
    return st


def run(state):
    c, s = state["c"], state["solver"]
    keep = (lambda v: v.to(torch.complex64)) if c["precision"] == "mixed" else (lambda v: v)
    if c["kind"] == "solve":
        call = bah.bah_solve_adjoint if c["adjoint"] else bah.bah_solve
        b = state["b"]
        x = state["x"] if c["host"] else torch.zeros_like(b)
        _, stats = call(s.ctx, b, x, c["sources"], 1e-14)
        return {"x": keep(x), "iters": np.array([q["iters"] for q in stats])}
    if c["kind"] == "precond":
        return {"z": keep(s.apply_preconditioner(state["x"]))}
    if c["kind"] == "operator":
        return {"y": s.apply_operator(state["x"]), "yh": s.apply_operator(state["x"], conj_transpose=True)}
    x, k = state["x"], c["sources"]
    adj = torch.empty_like(x)
    mis = torch.empty(k, dtype=torch.float64, device="cuda")
    g = torch.zeros((3,) + tuple(reversed(s.n)), dtype=torch.float64, device="cuda")
    bah.bah_misfit(s.ctx, x, state["d"], state["rec"], state["rec"].numel(), k, adj, mis)
    bah.bah_gradient(s.ctx, x, state["y"], k, g[0], g[1], g[2])
    return {"adjoint_sources": adj, "misfit": mis, "gradient": g}


def work(case):
    """Bytes and operations of one pass.  A solve step j (of a cycle of m) needs the flexible and
    the orthogonal basis vector written, the j + 1 basis vectors read for the projections and
    again for the update, the preconditioner's input and output, and the operator and stencil
    coefficients once; 8 operations per complex multiply-add of the Gram-Schmidt and about 250
    per unknown of a cycle and the operator."""
    c = _full(case)
    d = 3 if c["n3"] else 2
    cells = c["n1"] * c["n2"] * max(1, c["n3"])
    n, k = (d + 1) * cells, c["sources"]
    vb = 8 if c["precision"] == "mixed" else 16
    if c["kind"] == "operator":
        return {"bytes": 2.0 * k * n * 32 + 2.0 * cells * 56, "flops": 2.0 * k * cells * 84}
    if c["kind"] == "precond":
        return {"bytes": k * n * 32.0 + cells * (22.0 if vb == 8 else 96.0), "flops": k * n * 230.0}
    if c["kind"] == "gradient":
        return {"bytes": k * n * 48.0 + cells * 64.0, "flops": k * cells * 120.0}
    coef = cells * (56.0 + (22.0 if vb == 8 else 96.0))
    byts = flops = 0.0
    for q in range(c["steps"]):
        j = q % c["restart"]
        wide = k if c["block"] else 1      # columns each basis vector meets
        byts += k * n * (2.0 * vb + 16.0 * 3 + 2.0 * 16.0 * (j + 1)) + coef
        flops += k * n * (16.0 * (j + 1) * wide + 250.0)
        if j == c["restart"] - 1 or q == c["steps"] - 1:
            byts += k * n * (vb * (j + 1) + 64.0) + coef
            flops += k * n * (8.0 * (j + 1) * wide + 30.0)
    return {"bytes": byts + k * n * 32.0, "flops": flops}


# --------------------------------------------------------------------------
# the same outputs in 64 bits, from the equations
# --------------------------------------------------------------------------
def _operator(lam, mu, rho, gamma, omega, h, x, conj=False):
    """H [u; p] of Eq. 2.6 on a 2-D MAC grid (fields (n2, n1), x (k, 3, n2, n1)); the normal
    displacement and the tangential derivative terms vanish on the boundary."""
    h1, h2 = h
    rt = rho * (1.0 - 1j * gamma / omega)
    rt = rt.conj() if conj else rt
    u1, u2, p = x[:, 0].clone(), x[:, 1].clone(), x[:, 2]
    u1[:, :, 0] = 0
    u2[:, 0, :] = 0
    pad = torch.nn.functional.pad
    node = 0.25 * (mu[1:, 1:] + mu[1:, :-1] + mu[:-1, 1:] + mu[:-1, :-1])        # interior nodes

    def row(u, ax, ha, hb):
        t = (lambda a: a) if ax == 1 else (lambda a: a.transpose(-1, -2))
        u, m, nd, r, q = t(u), t(mu), t(node), t(rt), t(p)
        flux = m * (pad(u, (0, 1))[..., 1:] - u) / ha                            # at cells
        own = (flux[..., 1:] - flux[..., :-1]) / ha
        cross = pad(nd * (u[..., 1:, 1:] - u[..., :-1, 1:]) / hb, (0, 0, 1, 1))  # at nodes, zero outside
        cross = (cross[..., 1:, :] - cross[..., :-1, :]) / hb
        mass = omega * omega * 0.5 * (r[..., 1:] + r[..., :-1]) * u[..., 1:]
        return t(pad(-own - cross - mass + (q[..., 1:] - q[..., :-1]) / ha, (1, 0)))

    div = (pad(u1, (0, 1))[..., 1:] - u1) / h1 + (pad(u2, (0, 0, 0, 1))[..., 1:, :] - u2) / h2
    return torch.stack([row(u1, 1, h1, h2), row(u2, 0, h2, h1), -div - p / (lam + mu)], 1)


def exact(case, seed):
    """The outputs in 64 bits where they follow from the equations in a few lines.  A solve's
    iterate depends on the rounded multigrid hierarchy that the library builds, and so does the
    preconditioner's output: those have no value here."""
    c = _full(case)
    if c["kind"] not in ("operator", "gradient"):
        return None
    prob = _problem(c, seed)
    m = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (prob.lam, prob.mu, prob.rho, prob.gamma)]
    k = c["sources"]
    x = _fields(c, prob, seed, k)
    if c["kind"] == "operator":
        return {"y": _operator(*m, prob.omega, prob.h, x), "yh": _operator(*m, prob.omega, prob.h, x, True)}
    y = _fields(c, prob, seed + 1000003, k)
    rec = torch.from_numpy(receiver_indices(prob.n, max(1, prob.meta["abc"]))).cuda().long()
    d = torch.randn((k, len(rec)), dtype=torch.complex128, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(seed + 7))
    r = x.reshape(k, -1)[:, rec] - d
    adj = torch.zeros_like(x).reshape(k, -1)
    adj[:, rec] = r
    for a in m[:3]:
        a.requires_grad_(True)
    g = torch.zeros((3,) + prob.shape, dtype=torch.float64, device="cuda")
    for s in range(k):
        hx = _operator(*m, prob.omega, prob.h, x[s:s + 1])
        val = -(y[s:s + 1].conj() * hx).sum().real
        for q, ga in enumerate(torch.autograd.grad(val, m[:3])):
            g[q] += ga
    return {"adjoint_sources": adj.reshape(x.shape), "misfit": 0.5 * (r.real ** 2 + r.imag ** 2).sum(1), "gradient": g}
