"""What is timed of this package: time steps, gradients, the truncation's
backward and observables through the public calls a program makes.

A case is a dict of plain values with a "kind":
  step     one Heun or midpoint step of one PDF and its samples at probe points
           (or the whole dense PDF on a small grid): the stepping loop of a run
           that is watched while it goes
  batch    qtt_step_many over PDFs of uneven grid, bond and coefficients
  grad     the mean product J and its gradient through autograd.MeanProduct
  vjp      the backward of the bond truncation
  observe  the observables of a PDF: probe points, the mean fields over x, the
           scalars

The FP64 form's results are kept as they come, in 64 bits.  A program that
steps in a reduced form keeps its samples in 32 bits: the form's products
carry 24 (fp32) or 31 (bf16x10) bits of the row maxima, its factorisations
are float ones, and two processes already differ by 1e-7 to 1e-5 of f after
one step, since the tile and split choices are timed.  The FP64 steps
truncate at 1e-5 of the largest singular value: the right Grams resolve a
spectrum down to 1.5e-8 of it, and a cut made in that noise is arbitrary.
The tf32 and bf16x3 forms (1e-2 and 1e-4 per step) are not timed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2407_09169_gb300 as q
import workload
from paper_2407_09169_gb300.autograd import MeanProduct

TAU = 2.0 * math.pi


def listed():
    return [
        # untruncated FP64 on the smallest grid of the tests: the parity run beside the
        # finite-difference solver; every product is tiny, the step is its launches
        dict(name="exact fp64 2^2", kind="step", bits="2,2,2,2,2", chi=32, form="fp64", exact=True, flow=0, rk=0,
             sgs=False, dense=True, points=0),
        # the 2^20-cell workload in plain FP64, read back whole for the comparison with the solver
        dict(name="small fp64 chi 32", kind="step", bits="4,4,4,4,4", chi=32, form="fp64", exact=False, flow=0, rk=0,
             sgs=False, dense=True, points=0),
        # the paper's jet through a vortex with the subgrid closures on (fields for gamma and Omega), untruncated:
        # their sum's rank is above every sketch here, and a truncated step follows the last bit by 1e-8
        dict(name="exact fp64 sgs paper flow", kind="step", bits="2,2,3,2,3", chi=64, form="fp64", exact=True, flow=1,
             rk=0, sgs=True, dense=True, points=0),
        # the 2^30-cell workload in plain FP64 and in the fp32 form that is compared with it
        dict(name="medium fp64 chi 64", kind="step", bits="6,6,6,6,6", chi=64, form="fp64", exact=False, flow=0, rk=0,
             sgs=False, dense=False, points=512),
        dict(name="medium fp32 chi 64", kind="step", bits="6,6,6,6,6", chi=64, form="fp32", exact=False, flow=0, rk=0,
             sgs=False, dense=False, points=512),
        # a grid of unequal dimensions at an odd chi, the paper's flow, midpoint rule, the accurate tensor-core form
        dict(name="ragged bf16x10 chi 77", kind="step", bits="6,5,7,6,5", chi=77, form="bf16x10", exact=False, flow=1,
             rk=1, sgs=False, dense=False, points=512),
        # the 2^40-cell workload in the form that the benchmark steps
        dict(name="large bf16x10 chi 128", kind="step", bits="8,8,8,8,8", chi=128, form="bf16x10", exact=False, flow=0,
             rk=0, sgs=False, dense=False, points=512),
        # independent PDFs of the batched configuration's grids and bonds advanced together
        dict(name="batch of 12 bf16x10", kind="batch", n=12, form="bf16x10", steps=4, points=64),
        # a gradient step of a fit of the coefficients and amplitudes, on the grid that the oracle checks
        dict(name="gradient fp64 chi 32", kind="grad", bits=4, chi=32, steps=2, ckpt=1, icmodes=16),
        # the truncation's backward at the small and the large workload's sizes
        dict(name="truncation vjp 20 sites", kind="vjp", sites=20, bond=40, chi=32, ybond=32, eps=1e-6),
        dict(name="truncation vjp 40 sites", kind="vjp", sites=40, bond=136, chi=128, ybond=128, eps=0.0),
        # what is read from a stored PDF of the 2^30-cell grid for a figure
        dict(name="observe chi 64", kind="observe", bits="6,6,6,6,6", chi=64, points=4096, means=True),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "vjp", "vjp", "observe", "grad", "exact", "batch"])
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    if kind == "exact":  # at most 12 sites: the centre bond doubles with every second site
        while True:
            b = [rng.randint(1, 3) for _ in range(5)]
            if 8 <= sum(b) <= 12:
                break
        return dict(kind="step", bits=",".join(map(str, b)), chi=2 ** (sum(b) // 2), form="fp64", exact=True,
                    flow=rng.randint(0, 1), rk=rng.randint(0, 1), sgs=rng.random() < 0.3, dense=True, points=0)
    if kind == "step":
        form = rng.choice(["fp64", "fp32", "bf16x10", "bf16x10"])
        if form == "fp64":
            b, chi = [rng.randint(3, 6) for _ in range(5)], log(16, 64)
        elif form == "fp32":  # the batched configuration's smaller half: cubes
            b, chi = [rng.randint(4, 6)] * 5, log(16, 64)
        else:
            b, chi = [rng.randint(4, 8) for _ in range(5)], log(16, 128)
        return dict(kind="step", bits=",".join(map(str, b)), chi=chi, form=form, exact=False,
                    flow=rng.randint(0, 1), rk=rng.randint(0, 1) if form != "fp32" else 0, sgs=False, dense=False,
                    points=log(32, 1024))
    if kind == "vjp":
        chi = log(8, 128)
        return dict(kind="vjp", sites=rng.randint(6, 40), bond=chi + rng.randint(0, 16), chi=chi, ybond=log(8, 128),
                    eps=rng.choice([0.0, 1e-6]))
    if kind == "grad":
        return dict(kind="grad", bits=rng.randint(3, 4), chi=log(16, 32), steps=rng.randint(1, 3),
                    ckpt=rng.randint(0, 2), icmodes=rng.randint(1, 16))
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(2, 10), form="bf16x10", steps=rng.randint(1, 2), points=log(16, 128))
    b = [rng.randint(3, 6) for _ in range(5)]
    return dict(kind="observe", bits=",".join(map(str, b)), chi=log(16, 128), points=log(64, 4096),
                means=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs
def _bits(case):
    return [int(b) for b in str(case["bits"]).split(",")]


def _params(case, seed):
    """Parameters of one PDF: the workloads' coefficients, modes drawn from the seed."""
    bits = _bits(case)
    small = {"bits": bits[0], "chi_max": case["chi"], "steps": 1}
    if case.get("flow", 0) == 1:
        p = workload.make_paper_params(bits=bits[0], chi=case["chi"], seed=seed, precision=case.get("form", "fp64"),
                                       umodes=workload.draw_velocity_modes(seed))
    else:
        p = workload.make_params(small, seed=seed, precision=case.get("form", "fp64"))
    p["bits"] = bits
    p["rk_variant"] = case.get("rk", 0)
    if case.get("exact"):
        p.update(exact=1, svd_rel_tol=0.0, chi_max=2 ** (sum(bits) // 2))
    elif case.get("form") == "fp64":
        p["svd_rel_tol"] = 1e-5
    if case.get("sgs"):
        p["sgs"] = 1
    p["dt"] = workload.cfl_dt(bits, p["omega"], p["da"], p["gamma"], p["d_phi"], workload.velocity_bound(p))
    return p


def _probe(p, n, seed):
    """n multi-indices [n, 5] where the PDF has its mass: composition near one of
    the two centres, x uniform."""
    rng = np.random.default_rng([seed, 77])
    M = [2 ** b for b in p["bits"]]
    hi = rng.random(n) < 0.5
    c = np.where(hi[:, None], np.array(p["ic_c_hi"]), np.array(p["ic_c_lo"]))
    phi = np.abs(c + 2.0 * p["ic_sigma"] * rng.standard_normal((n, 2)))
    phi = np.where(phi > 1.0, 2.0 - phi, phi).clip(0.0, 1.0)
    idx = [np.minimum((phi[:, a] * M[a]).astype(np.int64), M[a] - 1) for a in range(2)]
    idx += [rng.integers(0, M[d], n) for d in range(2, 5)]
    return np.stack(idx, 1)


def _flags(idx, bits):
    """The 0/1 index bits of qtt_observe(QTT_OBS_POINTS), most significant first."""
    cols = [(idx[:, d] >> (bits[d] - 1 - k)) & 1 for d in range(5) for k in range(bits[d])]
    return np.ascontiguousarray(np.stack(cols, 1).astype(np.float64).ravel())


def _batch_params(case, seed):
    """Da log-uniform in [0.1, 10], Omega uniform in [0.5, 2]; the grids and bonds
    of the batched configuration, each pair in turn."""
    rng = np.random.default_rng([seed, 5])
    out = []
    for i in range(case["n"]):
        da, om = float(10.0 ** rng.uniform(-1, 1)), float(rng.uniform(0.5, 2.0))
        w = {"bits": (5, 6, 7)[i % 3], "chi_max": (16, 32, 64, 96)[i % 4], "steps": 1}
        out.append(workload.make_params(w, seed=seed * 100 + i, precision=case["form"], da=da, omega=om,
                                        d_phi=4e-3 * om))
    return out


def _theta(case, seed):
    rng = np.random.default_rng([seed, 9])
    p = workload.make_params({"bits": case["bits"], "chi_max": case["chi"], "steps": 1}, seed=seed)
    p["svd_rel_tol"] = 1e-6
    p["icmodes"] = workload.draw_ic_modes(seed, case["icmodes"])
    v = [rng.uniform(0.8, 1.2), rng.uniform(0.8, 1.2), rng.uniform(0.8e-2, 1.2e-2)]
    v += list(rng.uniform(0.05, 0.15, len(p["umodes"]))) + list(rng.uniform(-0.05, 0.05, case["icmodes"]))
    return p, torch.tensor(v, dtype=torch.float32)


def _vjp_bonds(case):
    N = case["sites"]
    r = [min(2 ** min(n, N - n), case["bond"]) for n in range(N + 1)]
    s = [min(2 ** min(n, N - n), case["ybond"]) for n in range(N + 1)]
    return r, s


def _vjp_trains(case, seed):
    """X in the form the zip-up leaves (cores 0 .. N-2 left-orthonormal): random
    isometries, and where the bond shrinks towards the end orthogonal matrices
    with weights w, w' on the two values of the site (w^2 + w'^2 = 2), so that
    the right Grams' spectra decay over a few decades and stay above rounding.
    The cotangent is a Gaussian train, as large as makes the cut cores order one.
    Everything is drawn on the host."""
    rng = np.random.default_rng([seed, 3])
    N, (r, s) = case["sites"], _vjp_bonds(case)
    cores = []
    for n in range(N - 1):
        a, b = r[n], r[n + 1]
        if a >= 2 * b:
            U = np.linalg.qr(rng.standard_normal((a, 2 * b)))[0].reshape(a, 2, b)
            t = rng.uniform(0.1, 0.6, b)
            cores.append(U * np.sqrt(np.stack([1.0 + t, 1.0 - t]))[None] / math.sqrt(2.0))
        else:
            cores.append(np.linalg.qr(rng.standard_normal((2 * a, b)))[0].reshape(a, 2, b))
    cores.append(np.array([[1.0, 0.3], [-0.2, 0.7]])[: r[N - 1]].reshape(r[N - 1], 2, 1) * rng.uniform(0.8, 1.2))
    y = [rng.standard_normal((s[n], 2, s[n + 1])) / math.sqrt(2.0 * s[n]) for n in range(N)]
    y[0] *= 0.25 * case["bond"] ** 2
    return cores, y


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step" or kind == "observe":
        p = _params(case, seed)
        if kind == "observe":  # a stored PDF: its initial condition carries modes over x
            p["icmodes"] = _observe_modes(seed)
        ctx = q.qtt_init(p)
        idx = _probe(p, case["points"], seed) if case["points"] else None
        return dict(kind=kind, case=case, ctx=ctx, flags=_flags(idx, p["bits"]) if idx is not None else None)
    if kind == "batch":
        ps = _batch_params(case, seed)
        return dict(kind=kind, case=case, ctxs=[q.qtt_init(p) for p in ps],
                    flags=[_flags(_probe(p, case["points"], seed + i), p["bits"]) for i, p in enumerate(ps)])
    if kind == "grad":
        p, theta = _theta(case, seed)
        return dict(kind=kind, case=case, params=p, theta=theta.cuda().requires_grad_(True))
    cores, y = _vjp_trains(case, seed)
    r, s = _vjp_bonds(case)
    N = case["sites"]
    cap = sum((1 if n == 0 else 2 * r[n]) * 2 * (1 if n == N - 1 else 2 * r[n + 1]) for n in range(N))
    flat = lambda cs: torch.from_numpy(np.concatenate([c.ravel() for c in cs])).cuda()  # noqa: E731
    return dict(kind=kind, case=case, r=r, s=s, x=flat(cores), y=flat(y), cap=cap,
                out=torch.empty(cap, dtype=torch.float64, device="cuda"))


def _observe_modes(seed):
    rng = np.random.default_rng([seed, 21])
    modes = workload.draw_ic_modes(seed, 8)
    for m in modes:
        m["amp"] = float(rng.uniform(0.02, 0.08))
    return modes


def _sample(ctx, flags, form):
    v = ctx.observe(q.OBS_POINTS, out=flags.copy())
    return v.copy() if form == "fp64" else v.astype(np.float32)


def run(state):
    case, kind = state["case"], state["kind"]
    if kind == "step":
        ctx = state["ctx"]
        ctx.step(1)
        return ctx.observe(q.OBS_DENSE) if case["dense"] else _sample(ctx, state["flags"], case["form"])
    if kind == "batch":
        q.qtt_step_many(state["ctxs"], case["steps"])
        return np.concatenate([_sample(c, f, case["form"]) for c, f in zip(state["ctxs"], state["flags"])])
    if kind == "grad":
        theta = state["theta"]
        theta.grad = None
        J = MeanProduct.apply(theta, state["params"], case["steps"], case["ckpt"])
        J.backward()
        return {"J": J.detach(), "grad": theta.grad}
    if kind == "vjp":
        _, kept = q.qtt_truncate_vjp(state["r"], state["x"], state["s"], state["y"], case["chi"], 1e-7, case["eps"],
                                     state["out"], state["cap"])
        return {"xbar": state["out"], "kept": np.array(kept, dtype=np.int64)}
    ctx = state["ctx"]
    out = {"points": _sample(ctx, state["flags"], "fp64"), "scalars": ctx.observe(q.OBS_SCALARS)}
    if case["means"]:
        out["means"] = ctx.observe(q.OBS_MEANS)
    return out


# -------------------------------------------------------------------- work
def _profile(bits, chi):
    N = sum(bits)
    return [min(2 ** min(n, N - n), chi) for n in range(N + 1)]


def _step_flops(bits, chi, exact, sgs=False):
    """2 m n k of one step's contractions: per stage, site and term, the sketch
    and the projection of an operator (bond ~16, the mixing term's on x the
    state's own bond) times the state, and the factorisations."""
    D, kphi, tot = _profile(bits, chi), bits[0] + bits[1], 0.0
    ell = [min(2 ** min(n, sum(bits) - n), chi + (0 if exact else 8)) for n in range(len(D))]
    for n in range(sum(bits)):
        a, b, la, lb = D[n], D[n + 1], ell[n], ell[n + 1]
        for lin in (True, False):
            wa, wb = (min(16, 4 ** n), min(16, 4 ** (sum(bits) - n - 1))) if lin or n < kphi else (a, b)
            if sgs and not lin and n >= kphi:  # times the mixing rate's bond, full on these grids
                wa, wb = (a * 2 ** min(n - kphi, sum(bits) - n), b * 2 ** min(n + 1 - kphi, sum(bits) - n - 1))
            env = 2 * wb * b * 2 * la * lb + 2 * wb * a * b * 2 * la + 2 * wa * wb * a * 2 * la
            tot += env if exact else 2 * env
        tot += 0 if exact else 8.0 * la * lb * lb + 10.0 * lb ** 3
    return 2.0 * tot  # two stages


def _state_bytes(bits, chi):
    D = _profile(bits, chi)
    return 8.0 * sum(D[n] * 2 * D[n + 1] for n in range(sum(bits)))


def work(case):
    kind = case["kind"]
    if kind == "step":
        b = _bits(case)
        out = 8.0 * (2 ** sum(b) if case["dense"] else case["points"] * (1 + sum(b)))
        extra = case["points"] * _state_bytes(b, case["chi"]) / 8
        if case["dense"]:
            extra = 2.0 * 2 ** sum(b) * case["chi"] ** 0.5
        return {"bytes": 2 * _state_bytes(b, case["chi"]) + out,
                "flops": _step_flops(b, case["chi"], case["exact"], case["sgs"]) + extra}
    if kind == "batch":
        fl = by = 0.0
        for i in range(case["n"]):
            b, chi = [(5, 6, 7)[i % 3]] * 5, (16, 32, 64, 96)[i % 4]
            fl += case["steps"] * _step_flops(b, chi, False) + case["points"] * _state_bytes(b, chi) / 8
            by += 2 * _state_bytes(b, chi) * case["steps"] + 8.0 * case["points"]
        return {"bytes": by, "flops": fl}
    if kind == "grad":  # a step forward, its recompute and a backward step of three terms
        b = [case["bits"]] * 5
        again = 2 if case["ckpt"] and case["ckpt"] < case["steps"] else 1
        return {"bytes": 6 * case["steps"] * _state_bytes(b, case["chi"]),
                "flops": case["steps"] * (1 + again + 3) * _step_flops(b, case["chi"], False)}
    if kind == "vjp":
        (r, s), fl, by = _vjp_bonds(case), 0.0, 0.0
        for n in range(case["sites"]):
            a, b, sa, sb = r[n], r[n + 1], s[n], s[n + 1]
            fl += 2.0 * (2 * a * b * b + a * a * 2 * b)          # right Gram
            fl += 2.0 * (a * sa * 2 * sb + 2 * a * b * sb + b * b * sb)  # left environment
            fl += 2.0 * (2 * a * b * b + 2 * sa * sb * b + sa * a * 2 * b)  # right environment
            fl += 2.0 * (2 * a * sb * b + 4 * 2 * a * b * b) + 9.0 * b ** 3  # cut core, eigenpairs
            by += 8.0 * (2 * a * b + 2 * sa * sb + 8 * a * b)
        return {"bytes": by, "flops": fl}
    b = _bits(case)
    D, N, kphi = _profile(b, case["chi"]), sum(b), b[0] + b[1]
    fl = 2.0 * case["points"] * sum(D[n] * D[n + 1] for n in range(N))
    fl += 2.0 * 6 * sum(2 * D[n] * D[n + 1] for n in range(kphi))
    fl += 2.0 * sum(2 * D[n] * D[n + 1] * (D[n] + D[n + 1]) for n in range(N))
    by = _state_bytes(b, case["chi"]) + 8.0 * case["points"] * (1 + N)
    if case["means"]:
        by += 3 * 8.0 * 2 ** (N - kphi)
        fl += 3 * 2.0 * sum(2 ** (n - kphi) * 2 * D[n] * D[n + 1] for n in range(kphi, N))
    return {"bytes": by, "flops": fl}


# ------------------------------------------- 64-bit values in plain torch
def _grid(bits):
    M = [2 ** b for b in bits]
    ax = [(torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) / m for m in M[:2]]
    ax += [torch.arange(m, dtype=torch.float64, device="cuda") * (TAU / m) for m in M[2:]]
    return M, ax, [1.0 / m for m in M[:2]] + [TAU / m for m in M[2:]]


def _velocity(p, ax):
    X = torch.meshgrid(*ax[2:], indexing="ij")
    z = torch.zeros_like(X[0])
    u = [z.clone(), z.clone(), z.clone()]
    if p.get("flow", 0) == 1:
        jet = torch.exp(-((X[1] / TAU - 0.5) ** 2 + (X[2] / TAU - 0.5) ** 2) * 18.0)
        s, c = [torch.sin(2 * x) for x in X], [torch.cos(2 * x) for x in X]
        u = [p["u0"] * (c[0] * s[1] * s[2] - jet), p["u0"] * s[0] * c[1] * s[2], -2.0 * p["u0"] * s[0] * s[1] * c[2]]
    else:
        u[0] = u[0] + p["shear_amp"] * torch.tanh(X[1] - math.pi)
    for m in p["umodes"]:
        k = m["k"]
        u[m["comp"]] = u[m["comp"]] + m["amp"] * torch.sin(k[0] * X[0] + k[1] * X[1] + k[2] * X[2] + m["phase"])
    return u


def _blend(p, ax):
    """(Gaussian factors at the two centres, weight of the first over x, modulation over x)."""
    w, sig = p["ic_blend_width"], p["ic_sigma"]
    g = []
    for c in (p["ic_c_hi"], p["ic_c_lo"]):
        f = [torch.exp(-(ax[a] - c[a]) ** 2 / (2.0 * sig * sig)) for a in range(2)]
        g.append([v / (v.sum() / v.numel()) for v in f])
    X = torch.meshgrid(*ax[2:], indexing="ij")
    if p.get("ic_kind", 0) == 1:
        wx = 0.5 * (torch.tanh((X[0] - 0.5 * math.pi) / w) - torch.tanh((X[0] - 1.5 * math.pi) / w))
    else:
        wx = 0.5 * (1.0 + torch.tanh((X[1] - math.pi) / w))
    mod = torch.ones_like(wx)
    for m in p.get("icmodes", []):
        k = m["k"]
        mod = mod + m["amp"] * torch.cos(k[0] * X[0] + k[1] * X[1] + k[2] * X[2] + m["phase"])
    return g, wx, mod


def _initial(p, ax):
    g, wx, mod = _blend(p, ax)
    hi, lo = [torch.outer(v[0], v[1])[:, :, None, None, None] for v in g]
    return hi * (wx * mod) + lo * ((1.0 - wx) * mod)


def _ghost(f, d, sign):
    n = f.shape[d]
    return torch.cat([sign * f.narrow(d, 0, 1), f, sign * f.narrow(d, n - 1, 1)], d)


def _rhs(f, p, ax, h, u):
    M = f.shape
    gam, om = p["gamma"], p["omega"]
    if p.get("sgs"):
        width = p.get("delta_cells", 3.0) * (h[2] * h[3] * h[4]) ** (1.0 / 3.0)
        d1 = lambda v, j: (torch.roll(v, -1, j) - torch.roll(v, 1, j)) / (2.0 * h[2 + j])  # noqa: E731
        s2 = sum((d1(u[i], j) + d1(u[j], i)) ** 2 for i in range(3) for j in range(3))
        gam = p["gamma"] + p.get("c_s", 0.11) * 0.5 * width ** 2 * torch.sqrt(s2)
        om = p.get("c_omega", 0.5) * gam / width ** 2
    out = torch.zeros_like(f)
    for i in range(3):
        a = 2 + i
        up, dn = torch.roll(f, -1, a), torch.roll(f, 1, a)
        out = out - u[i] * ((up - dn) / (2.0 * h[a]))
        if p.get("sgs"):
            face = 0.5 * (gam + torch.roll(gam, -1, i))
            out = out + (face * (up - f) - torch.roll(face, 1, i) * (f - dn)) / h[a] ** 2
        else:
            out = out + gam * ((up - 2.0 * f + dn) / h[a] ** 2)
        del up, dn
    P = [ax[0].view(-1, 1, 1, 1, 1), ax[1].view(1, -1, 1, 1, 1)]
    cell = h[0] * h[1]
    for a in range(2):
        mean = cell * (P[a] * f).sum((0, 1))
        g = _ghost((om * (P[a] - mean) + p["da"] * P[0] * P[1]) * f, a, -1.0)
        out = out + (g.narrow(a, 2, M[a]) - g.narrow(a, 0, M[a])) / (2.0 * h[a])
        del g
        e = _ghost(f, a, 1.0)
        out = out + p["d_phi"] * (e.narrow(a, 2, M[a]) - 2.0 * f + e.narrow(a, 0, M[a])) / h[a] ** 2
        del e
    return out


def _dense_step(f, p, ax, h, u):
    if p.get("rk_variant", 0) == 1:
        return f + p["dt"] * _rhs(f + 0.5 * p["dt"] * _rhs(f, p, ax, h, u), p, ax, h, u)
    fs = f + p["dt"] * _rhs(f, p, ax, h, u)
    return 0.5 * (f + fs + p["dt"] * _rhs(fs, p, ax, h, u))


def _dense_points(p, n, idx):
    _, ax, h = _grid(p["bits"])
    u = _velocity(p, ax)
    f = _initial(p, ax)
    for _ in range(n):
        f = _dense_step(f, p, ax, h, u)
    if idx is None:
        return f.reshape(-1).cpu().numpy()
    i = torch.from_numpy(idx).cuda()
    return f[i[:, 0], i[:, 1], i[:, 2], i[:, 3], i[:, 4]].cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        p = _params(case, seed)
        if sum(p["bits"]) > 30:  # over 2^30 cells the dense grid does not fit beside its temporaries
            return None
        idx = _probe(p, case["points"], seed) if case["points"] else None
        v = _dense_points(p, 1, idx)
        return v if case["form"] == "fp64" else v.astype(np.float32)
    if kind == "batch":
        return None  # grids of up to 2^35 cells
    if kind == "grad":
        return _exact_grad(case, seed)
    if kind == "vjp":
        return _exact_vjp(case, seed)
    return _exact_observe(case, seed)


def _exact_grad(case, seed):
    """J and its gradient by reverse differentiation of the dense steps."""
    p, theta = _theta(case, seed)
    t = theta.double().cuda().requires_grad_(True)
    nu = len(p["umodes"])
    p = dict(p, omega=t[0], da=t[1], gamma=t[2], umodes=[dict(m, amp=t[3 + i]) for i, m in enumerate(p["umodes"])],
             icmodes=[dict(m, amp=t[3 + nu + i]) for i, m in enumerate(p["icmodes"])])
    _, ax, h = _grid(p["bits"])
    u, f = _velocity(p, ax), _initial(p, ax)
    for _ in range(case["steps"]):
        f = _dense_step(f, p, ax, h, u)
    one = 1.0 - ax[0].view(-1, 1, 1, 1, 1) - ax[1].view(1, -1, 1, 1, 1)
    J = (one * f).sum() * (h[0] * h[1] / (f.shape[2] * f.shape[3] * f.shape[4]))
    J.backward()
    return {"J": J.detach().float(), "grad": t.grad.float()}


def _exact_vjp(case, seed):
    """(dT/dX)^T ybar of T(X) = Pi_1 .. Pi_{N-1} X as a train: the part with the
    projectors fixed, and per cut the derivative of the projector through the
    null space (weights 1 / lambda) and through the gaps (1 / (lambda_i -
    lambda_j), kept i and dropped j; Lorentzian for eps > 0)."""
    cores, ys = _vjp_trains(case, seed)
    N, (r, s), eps = case["sites"], _vjp_bonds(case), case["eps"]
    Q = [torch.from_numpy(c).cuda() for c in cores]
    Y = [torch.from_numpy(c).cuda() for c in ys]
    wgt = lambda d: d / (d * d + eps * eps)  # noqa: E731
    G = [None] * N
    G[N - 1] = Q[N - 1].reshape(r[N - 1], 2) @ Q[N - 1].reshape(r[N - 1], 2).T
    for n in range(N - 1, 1, -1):
        G[n - 1] = torch.einsum("aib,bc,dic->ad", Q[n - 1], G[n], Q[n - 1])
    V, lam, k, P = [None] * N, [None] * N, [0] * N, [None] * N
    for n in range(1, N):
        w, U = torch.linalg.eigh(G[n].cpu())
        lam[n], V[n] = w.flip(0).cuda(), U.flip(1).cuda()
        k[n] = int(min(case["chi"], int((lam[n] > 1e-14 * lam[n][0]).sum())))
        P[n] = V[n][:, : k[n]] @ V[n][:, : k[n]].T
    Qm = [None] + [Q[n - 1].reshape(-1, r[n]) for n in range(1, N)]
    e, Yh = [torch.ones(1, 1, dtype=torch.float64, device="cuda")], [None] * N
    for n in range(1, N):
        Yh[n] = torch.einsum("as,sib->aib", e[-1], Y[n - 1]).reshape(-1, s[n])
        e.append(P[n] @ (Qm[n].T @ Yh[n]))
    R = [None] * N
    R[N - 1] = Y[N - 1].reshape(s[N - 1], 2) @ Q[N - 1].reshape(r[N - 1], 2).T
    for n in range(N - 1, 1, -1):
        R[n - 1] = torch.einsum("sit,tb,aib->sa", Y[n - 1], R[n], (Qm[n] @ P[n]).reshape(r[n - 1], 2, r[n]))
    out = []
    for n in range(1, N):
        g, kk = Yh[n] @ R[n], k[n]
        VK, VD, lk, ld = V[n][:, :kk], V[n][:, kk:], lam[n][:kk], lam[n][kk:]
        A = (VK * wgt(lk)) @ VK.T
        S = Qm[n].T @ g
        Gam = VD @ (wgt(lk[None, :] - ld[:, None]) * (VD.T @ (S + S.T) @ VK)) @ VK.T
        d = ((g - Qm[n] @ S) @ A + Qm[n] @ (Gam + Gam.T)).reshape(r[n - 1], 2, r[n])
        c = torch.cat([Q[n - 1], d], 2)
        if n > 1:
            c = torch.cat([c, torch.cat([torch.zeros_like(d), Q[n - 1]], 2)], 0)
        out.append(c.reshape(-1))
    last = torch.einsum("as,sib->aib", e[N - 1], Y[N - 1])
    out.append(torch.cat([last, Q[N - 1]], 0).reshape(-1))
    return {"xbar": torch.cat(out), "kept": np.array(k[1:], dtype=np.int64)}


def _exact_observe(case, seed):
    """The observables of the initial PDF hi(phi) a(x) + lo(phi) b(x) from its factors."""
    p = _params(case, seed)
    p["icmodes"] = _observe_modes(seed)
    _, ax, h = _grid(p["bits"])
    g, wx, mod = _blend(p, ax)
    a, b = wx * mod, (1.0 - wx) * mod
    idx = torch.from_numpy(_probe(p, case["points"], seed)).cuda()
    at = lambda v: v[idx[:, 2], idx[:, 3], idx[:, 4]]  # noqa: E731
    phi = lambda c: g[c][0][idx[:, 0]] * g[c][1][idx[:, 1]]  # noqa: E731
    pts = phi(0) * at(a) + phi(1) * at(b)
    m = lambda c, i, w: float((w * g[c][i]).sum() * h[i])  # noqa: E731  one-dimensional moments
    one = [torch.ones_like(ax[0]), torch.ones_like(ax[1])]
    mom = lambda w0, w1: [m(c, 0, w0) * m(c, 1, w1) for c in range(2)]  # noqa: E731
    field = lambda v: v[0] * a + v[1] * b  # noqa: E731
    n0, f1, f2 = field(mom(*one)), field(mom(ax[0], one[1])), field(mom(one[0], ax[1]))
    mean = lambda v: float(v.mean())  # noqa: E731
    p11, p22 = mean(field(mom(ax[0] ** 2, one[1]))), mean(field(mom(one[0], ax[1] ** 2)))
    p12 = mean(field(mom(ax[0], ax[1])))
    m12 = float((f1 * f2).mean())
    gg = lambda c, d: float((g[c][0] * g[d][0]).sum() * (g[c][1] * g[d][1]).sum())  # noqa: E731
    n2 = gg(0, 0) * float((a * a).sum()) + 2.0 * gg(0, 1) * float((a * b).sum()) + gg(1, 1) * float((b * b).sum())
    sc = [0.0, mean(n0), mean(f1), mean(f2), p11, p22, p12, m12 - mean(f1) * mean(f2), p12 - m12,
          mean(n0) - mean(f1) - mean(f2), 0.0, 0.0, n2]
    out = {"points": pts.cpu().numpy(), "scalars": np.array(sc)}
    if case["means"]:
        out["means"] = torch.cat([n0.reshape(-1), f1.reshape(-1), f2.reshape(-1)]).cpu().numpy()
    return out
