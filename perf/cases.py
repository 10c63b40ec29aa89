"""The performance cases of this framework: what a program does with it, through its public entry points.

A program holds a plan, a problem (its conductivity on the GPU), a workspace and a state, and advances the
state by some steps; it differentiates such a run; it advances many small problems in one launch; or it
integrates the Brusselator.  Every pass starts from the same initial state, which it copies into the state
that the call advances in place.

Sizes: the workload recipes of ``bench.py`` and ``bench_workloads.py`` (1D heat N = 256, 2D variable conductivity
2048^2 with s = 64, 3D kappa(u) = 1 + u^2.5 on 256^3 with s = 32, the 1024^2 adjoint with s = 100 and a checkpoint
every 8 steps, batches of uneven problems, the 200^2 Brusselator to t = 1 and its 2048^2 grid), and the ragged
Dirichlet grids that the tests use, at sizes between those.  The step is 0.9 beta / rho throughout.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

CFL = 0.9
STATE = {"fp64": torch.float64, "fp32": torch.float32, "mixed": torch.float64, "dfloat": torch.float64}
KAPPA = {"fp64": torch.float64, "fp32": torch.float32, "mixed": torch.float32, "dfloat": torch.float32}
# flops of one cell and stage: neighbour differences, fluxes, complex update (and kappa(W), the reaction, or
# the adjoint's transposed stencil and face sensitivities beside the forward stage)
FLOPS = {"heat1d": 18, "step2d": 26, "batched2d": 26, "step3d_field": 36, "step3d_power": 95, "adjoint2d": 72, "bruss2d": 63}


def listed():
    return [
        # the smallest call: a 1D rod, 87 steps of 16 stages in one call, bound by latency
        {"name": "heat1d_256_fp64", "kind": "heat1d", "nx": 256, "s": 16, "steps": 87, "prec": "fp64", "bc": "dirichlet"},
        # a small 2D model at full precision: each stage is a few microseconds of work
        {"name": "step2d_256_fp64", "kind": "step2d", "nx": 256, "ny": 256, "s": 32, "steps": 10, "prec": "fp64", "bc": "periodic"},
        # the headline workload at full precision
        {"name": "step2d_2048_fp64", "kind": "step2d", "nx": 2048, "ny": 2048, "s": 64, "steps": 2, "prec": "fp64", "bc": "periodic"},
        # the same in single precision with the stage order that the precision policy takes for it
        {"name": "step2d_2048_fp32", "kind": "step2d", "nx": 2048, "ny": 2048, "s": 64, "steps": 10, "prec": "fp32", "bc": "periodic"},
        # a grid as a user's domain gives it: odd sides, Dirichlet walls
        {"name": "step2d_1021x777_fp32", "kind": "step2d", "nx": 1021, "ny": 777, "s": 32, "steps": 10, "prec": "fp32", "bc": "dirichlet"},
        # where FP32 misses the tolerance in 2D, the policy takes the float-pair state
        {"name": "step2d_2048_dfloat", "kind": "step2d", "nx": 2048, "ny": 2048, "s": 64, "steps": 4, "prec": "dfloat", "bc": "periodic"},
        # nonlinear conduction in 3D
        {"name": "step3d_256_fp32", "kind": "step3d", "nx": 256, "ny": 256, "nz": 256, "s": 32, "steps": 1, "prec": "fp32", "bc": "dirichlet", "kappa": "power"},
        # where FP32 misses the tolerance for kappa(u), the policy takes the mixed precision; ragged box
        {"name": "step3d_121x150x97_mixed", "kind": "step3d", "nx": 121, "ny": 150, "nz": 97, "s": 16, "steps": 2, "prec": "mixed", "bc": "dirichlet", "kappa": "power"},
        # gradients with respect to the initial state and the conductivity (forward and backward)
        {"name": "adjoint2d_1024_fp32", "kind": "adjoint2d", "nx": 1024, "ny": 1024, "s": 100, "steps": 8, "ckpt": 8, "prec": "fp32", "bc": "periodic"},
        # a serving batch: many uneven problems in one launch
        {"name": "batched2d_32_fp32", "kind": "batched2d", "count": 32, "nmin": 64, "nmax": 1024, "steps": 2, "prec": "fp32", "bc": "periodic"},
        # the paper's demonstration problem, to t = 1
        {"name": "bruss2d_200_fp64", "kind": "bruss2d", "nx": 200, "ny": 200, "s": 16, "steps": 42, "prec": "fp64", "bc": "periodic"},
        # the same system on a large grid in single precision
        {"name": "bruss2d_2048_fp32", "kind": "bruss2d", "nx": 2048, "ny": 2048, "s": 16, "steps": 10, "prec": "fp32", "bc": "periodic"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes spread over the logarithm of the range, odd ones among them, and as many steps as a
    run of that size takes in a few milliseconds."""
    kind = rng.choice(["heat1d", "step2d", "step2d", "step2d", "step3d", "step3d", "adjoint2d", "batched2d", "bruss2d", "bruss2d"])
    c = {"kind": kind, "bc": rng.choice(["periodic", "dirichlet"])}
    if kind == "heat1d":
        c.update(nx=_log(rng, 64, 4096), s=rng.choice([8, 16, 32]), steps=rng.randint(20, 90), prec=rng.choice(["fp64", "fp32"]))
    elif kind == "step2d":
        c.update(nx=_log(rng, 64, 2048), ny=_log(rng, 64, 2048), s=rng.choice([16, 32, 64, 128]),
                 prec=rng.choice(["fp64", "fp64", "fp32", "fp32", "dfloat", "mixed"]))
        most = 5e8 if c["prec"] in ("fp64", "mixed") else 2.5e9
        c["steps"] = max(1, min(10, int(most / (c["nx"] * c["ny"] * c["s"]))))
    elif kind == "step3d":
        c.update(nx=_log(rng, 40, 250), ny=_log(rng, 40, 250), nz=_log(rng, 40, 250), s=rng.choice([8, 16, 32]),
                 prec=rng.choice(["fp64", "fp32", "mixed"]), kappa=rng.choice(["power", "power", "field"]))
        most = {"fp64": 6e7, "mixed": 2e8, "fp32": 5e8}[c["prec"]]
        c["steps"] = max(1, min(4, int(most / (c["nx"] * c["ny"] * c["nz"] * c["s"]))))
    elif kind == "adjoint2d":
        c.update(nx=_log(rng, 64, 1000), ny=_log(rng, 64, 1000), s=rng.choice([16, 32, 64]), steps=rng.randint(2, 8), ckpt=rng.choice([4, 8]),
                 prec=rng.choice(["fp64", "fp32"]))
        if c["prec"] == "fp64":
            c["steps"] = max(2, min(c["steps"], int(1.2e8 / (c["nx"] * c["ny"] * c["s"]))))
    elif kind == "batched2d":
        lo = _log(rng, 32, 200)
        c.update(count=rng.randint(4, 32), nmin=lo, nmax=_log(rng, 2 * lo, 1024), steps=rng.randint(1, 2), prec=rng.choice(["fp64", "fp32"]))
        if c["prec"] == "fp64":
            c.update(count=min(c["count"], 16), nmax=min(c["nmax"], 512), steps=1)
    else:
        c.update(nx=_log(rng, 64, 2048), ny=_log(rng, 64, 2048), s=rng.choice([8, 16, 32]), prec=rng.choice(["fp64", "fp32"]),
                 bc=rng.choice(["periodic", "neumann"]))
        most = 1.2e8 if c["prec"] == "fp64" else 7e8
        c["steps"] = max(1, min(20, int(most / (c["nx"] * c["ny"] * c["s"]))))
    return c


# ---- inputs -------------------------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _smooth(shape, ell, gen):
    """Gaussian random field of correlation length ell cells, mean 0 and standard deviation 1 (float64)."""
    xi = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    f2 = torch.zeros((), device="cuda", dtype=torch.float64)
    for ax, n in enumerate(shape):
        f = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) ** 2
        f2 = f2 + f.reshape([n if a == ax else 1 for a in range(len(shape))])
    g = torch.fft.ifftn(torch.fft.fftn(xi) * torch.exp(-2.0 * math.pi ** 2 * ell ** 2 * f2)).real
    g = g - g.mean()
    return (g / g.std()).contiguous()


def _unit(shape, ell, gen):
    g = _smooth(shape, ell, gen)
    return (g - g.min()) / (g.max() - g.min())


def _field2d(nx, ny, gen, prec):
    """Log-normal conductivity and a smooth state in [0, 1], as the 2D recipe has them."""
    side = max(nx, ny)
    kappa = torch.exp(0.5 * _smooth((ny, nx), 32.0 * side / 2048, gen)).to(KAPPA[prec])
    return kappa, _unit((ny, nx), 64.0 * side / 2048, gen).to(STATE[prec])


def _inputs(case, seed):
    """Inputs of a case as torch tensors on the GPU, from the seed alone."""
    gen, kind, prec = _gen(seed), case["kind"], case["prec"]
    if kind == "heat1d":
        n = case["nx"]
        amp = torch.randn(8, generator=gen, device="cuda", dtype=torch.float64)
        x = torch.arange(1, n + 1, device="cuda", dtype=torch.float64) / (n + 1)
        u = (amp[:, None] * torch.sin(math.pi * torch.arange(1, 9, device="cuda", dtype=torch.float64)[:, None] * x)).sum(0)
        return {"u": u.to(STATE[prec])}
    if kind in ("step2d", "adjoint2d"):
        kappa, u = _field2d(case["nx"], case["ny"], gen, prec)
        got = {"kappa": kappa, "u": u}
        if kind == "adjoint2d":
            got["target"] = _unit(tuple(u.shape), 64.0 * max(u.shape) / 2048, gen).to(STATE[prec])
        return got
    if kind == "step3d":
        shape = (case["nz"], case["ny"], case["nx"])
        if case["kappa"] == "field":
            ell = max(shape) / 64.0
            return {"kappa": torch.exp(0.5 * _smooth(shape, ell, gen)).to(KAPPA[prec]), "u": _unit(shape, 2 * ell, gen).to(STATE[prec])}
        # a hot spot of peak 2 with 1 % noise
        sigma, r2 = 20.0 * min(shape) / 256, torch.zeros((), device="cuda", dtype=torch.float64)
        for ax, n in enumerate(shape):
            i = torch.arange(n, device="cuda", dtype=torch.float64) - (n - 1) / 2.0
            r2 = r2 + (i * i).reshape([n if a == ax else 1 for a in range(3)])
        u = 2.0 * torch.exp(-r2 / (2.0 * sigma ** 2)) + 0.02 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
        return {"u": u.to(STATE[prec])}
    if kind == "batched2d":
        rng = np.random.default_rng(case["count"] * 1000 + case["nmax"])  # the sizes belong to the case, the fields to the seed
        got = []
        for _ in range(case["count"]):
            n, s = int(rng.integers(case["nmin"], case["nmax"] + 1)), int(rng.choice([16, 32, 64, 128]))
            kappa, u = _field2d(n, n, gen, prec)
            got.append({"kappa": kappa, "u": u, "s": s})
        return {"problems": got}
    nx, ny = case["nx"], case["ny"]
    dx = 1.0 / max(nx, ny)
    x = torch.arange(nx, device="cuda", dtype=torch.float64) / nx
    y = torch.arange(ny, device="cuda", dtype=torch.float64) / ny
    ell = max(nx, ny) / 32.0
    v = 1.0 + torch.sin(2 * math.pi * x)[None, :] + 0.1 * _smooth((ny, nx), ell, gen)
    w = 3.0 + torch.cos(2 * math.pi * y)[:, None] + 0.1 * _smooth((ny, nx), ell, gen)
    return {"v": v.to(STATE[prec]), "w": w.to(STATE[prec]), "dx": dx}


# ---- the method in 64 bits, in plain torch ---------------------------------------------------------


def _alpha(s):
    return 4.0 * (1.0 - 1.0 / (s * s)) / 3.0


def _beta(s):
    return 2.0 * (s * s - 1.0) / 3.0


def _shift(a, ax, step, bc, ghost):
    """Neighbour values of ``a`` along an axis: periodic wrap, or ``ghost`` outside ("edge": the cell's own)."""
    if bc == "periodic":
        return torch.roll(a, -step, ax)
    n = a.shape[ax]
    end = a.narrow(ax, n - 1 if step > 0 else 0, 1)
    out = end if ghost == "edge" else torch.full_like(end, ghost)
    return torch.cat([a.narrow(ax, 1, n - 1), out], ax) if step > 0 else torch.cat([out, a.narrow(ax, 0, n - 1)], ax)


def _faces(kappa, bc, ghost="edge"):
    return [(0.5 * (kappa + _shift(kappa, ax, -1, bc, ghost)), 0.5 * (kappa + _shift(kappa, ax, 1, bc, ghost))) for ax in range(kappa.dim())]


def _apply(w, faces, bc):
    """div(kappa grad w) with dx = 1 from face conductivities."""
    out = 0.0
    for ax, (lo, hi) in enumerate(faces):
        out = out + lo * (_shift(w, ax, -1, bc, 0.0) - w) + hi * (_shift(w, ax, 1, bc, 0.0) - w)
    return out


def _rho(faces):
    return float((2.0 * sum(lo + hi for lo, hi in faces)).max())


def _dt(s, rho):
    return CFL * _beta(s) / rho


def _linear_step(u, faces, bc, dt, s):
    """R(dt f) u for a linear f, R(z) = 1 - alpha/4 + (alpha/4) T_s(1 + 4 z / (s^2 alpha)), by the Chebyshev recurrence."""
    al = _alpha(s)
    c = 4.0 * dt / (s * s * al)
    t0, t1 = u, u + c * _apply(u, faces, bc)
    for _ in range(s - 1):
        t0, t1 = t1, 2.0 * (t1 + c * _apply(t1, faces, bc)) - t0
    return (1.0 - al / 4.0) * u + (al / 4.0) * t1


def _stages(s):
    """Complex step sizes in the paper's greedy stage order (its first pass, enough up to s = 32): for a nonlinear f the order counts."""
    al, m = _alpha(s), s // 2
    j = np.arange(s)
    z = np.cos((np.pi * (2 * j + 1) - 1j * np.arccosh(4.0 / al - 1.0)) / s)
    a = 1.0 / (m * m * al * (1.0 - z))
    a[m:] = np.conj(a[:m][::-1])
    k = np.arange(1, 16 * s + 1)
    logv = np.log(np.abs(1.0 + np.outer(a, -(1.0 - 1e-4) * _beta(s) * k / (16 * s))))
    left, placed, done = list(range(s)), [], np.zeros(16 * s)
    while left:
        cand = logv[left]
        e = np.maximum(done + cand, cand.sum(0) - cand)
        top = e.max(1)
        pick = left.pop(int(np.argmin(top + np.log(np.exp(e - top[:, None]).sum(1)))))
        placed.append(pick)
        done = done + logv[pick]
    return a[placed]


def _kappa_u(w):
    return 1.0 + w * w * torch.sqrt(w)


def _power_dt(u, bc, s):
    return _dt(s, _rho(_faces(_kappa_u(u.double()), bc, 1.0)))


def _bruss_dt(case, dx):
    return 1.0 / 42 * (case["s"] ** 2 - 1) / 255.0 * (dx * 200) ** 2  # the paper's run: 42 steps of 16 stages to t = 1 on 200^2


def _linear_dt(case, kappa, s):
    return _dt(s, _rho(_faces(kappa.double(), case["bc"])))


def exact(case, seed):
    inp, kind, bc = _inputs(case, seed), case["kind"], case["bc"]
    if kind == "heat1d":
        n, s = case["nx"], case["s"]
        h2 = (1.0 / (n + 1)) ** 2
        u, faces = inp["u"].double(), _faces(torch.ones(n, device="cuda", dtype=torch.float64), bc)
        for _ in range(case["steps"]):
            u = _linear_step(u, faces, bc, _dt(s, 4.0 / h2) / h2, s)
        return u
    if kind == "step2d" or (kind == "step3d" and case["kappa"] == "field"):
        u, faces = inp["u"].double(), _faces(inp["kappa"].double(), bc)
        for _ in range(case["steps"]):
            u = _linear_step(u, faces, bc, _dt(case["s"], _rho(faces)), case["s"])
        return u
    if kind == "step3d":
        dt, u = _power_dt(inp["u"], bc, case["s"]), inp["u"].double()
        for _ in range(case["steps"]):
            w = u.to(torch.complex128)
            for a in _stages(case["s"]):
                w = w + complex(dt * a) * _apply(w, _faces(_kappa_u(w), bc, 1.0), bc)
            u = w.real.contiguous()
        return u
    if kind == "adjoint2d":
        u0, kappa = inp["u"].double().requires_grad_(True), inp["kappa"].double().requires_grad_(True)
        dt = _linear_dt(case, inp["kappa"], case["s"])
        u = u0
        for _ in range(case["steps"]):
            u = checkpoint(lambda u, k: _linear_step(u, _faces(k, bc), bc, dt, case["s"]), u, kappa, use_reentrant=False)
        du, dk = torch.autograd.grad(((u - inp["target"].double()) ** 2).sum(), (u0, kappa))
        return {"u": u.detach(), "du0": du, "dkappa": dk}
    if kind == "batched2d":
        got = []
        for p in inp["problems"]:
            u, faces = p["u"].double(), _faces(p["kappa"].double(), bc)
            for _ in range(case["steps"]):
                u = _linear_step(u, faces, bc, _dt(p["s"], _rho(faces)), p["s"])
            got.append(u)
        return got
    dx, dt = inp["dx"], _bruss_dt(case, inp["dx"])
    wrap = "periodic" if bc == "periodic" else "neumann"
    lap = lambda a: (sum(_shift(a, ax, st, wrap, "edge") for ax in (0, 1) for st in (-1, 1)) - 4.0 * a) * (0.02 / (dx * dx))  # noqa: E731
    v, w = inp["v"].double(), inp["w"].double()
    for _ in range(case["steps"]):
        v, w = v.to(torch.complex128), w.to(torch.complex128)
        for a in _stages(case["s"]):
            r = v * v * w
            v, w = v + complex(dt * a) * (lap(v) + 1.0 - 4.0 * v + r), w + complex(dt * a) * (lap(w) + 3.0 * v - r)
        v, w = v.real.contiguous(), w.real.contiguous()
    return {"v": v, "w": w}


# ---- the framework's calls ---------------------------------------------------------------------------


def _plan(F, case, s, linear=True):
    # single precision on a fixed conductivity takes the Lebedev-Finogenov order, as the precision policy does
    return F.frkc2_plan(s, flags=F.PLAN_LEBEDEV if linear and case["prec"] == "fp32" else 0)


def prepare(case, seed):
    from paper_1702_03818_gb300 import frkc2 as F

    inp, kind, bc, prec = _inputs(case, seed), case["kind"], case["bc"], case["prec"]
    st = {"kind": kind, "F": F, "steps": case.get("steps")}

    def workspace(size):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        F.frkc2_workspace_reset(ws)
        return ws

    if kind in ("heat1d", "step2d", "step3d"):
        s, u0 = case["s"], inp["u"]
        linear = kind != "step3d" or case["kappa"] == "field"
        if kind == "heat1d":
            h = 1.0 / (case["nx"] + 1)
            prob = F.make_problem(1, (case["nx"],), h, bc, "const", prec, kappa_c=1.0)
            dt = _dt(s, 4.0 / (h * h))
        else:
            n = tuple(reversed(u0.shape))
            if linear:
                prob, dt = F.make_problem(len(n), n, 1.0, bc, "field", prec, kappa_field=inp["kappa"]), _linear_dt(case, inp["kappa"], s)
            else:
                prob, dt = F.make_problem(3, n, 1.0, bc, "power", prec, kappa_c=1.0, kappa_p=2.5), _power_dt(u0, bc, s)
        st.update(plan=_plan(F, case, s, linear), prob=prob, dt=dt, u0=u0, u=u0.clone(), ws=workspace(F.frkc2_workspace_size(prob)))
    elif kind == "adjoint2d":
        from paper_1702_03818_gb300.autograd import frkc2_steps

        st.update(steps_fn=frkc2_steps, plan=_plan(F, case, case["s"]), dt=_linear_dt(case, inp["kappa"], case["s"]), bc=bc, prec=prec, ckpt=case["ckpt"],
                  u0=inp["u"].requires_grad_(True), kappa=inp["kappa"].requires_grad_(True), target=inp["target"])
    elif kind == "batched2d":
        ps = inp["problems"]
        plans = {s: _plan(F, case, s) for s in sorted({p["s"] for p in ps})}
        pad = [-p["u"].numel() % 4 for p in ps]  # every state starts on a 16-byte boundary of one array
        u0 = torch.cat([x for p, k in zip(ps, pad) for x in (p["u"].reshape(-1), p["u"].new_zeros(k))])
        flat, views, at = u0.clone(), [], 0
        for p, k in zip(ps, pad):
            views.append(flat[at:at + p["u"].numel()].view(p["u"].shape))
            at += p["u"].numel() + k
        probs = [F.make_problem(2, tuple(reversed(p["u"].shape)), 1.0, bc, "field", prec, kappa_field=p["kappa"]) for p in ps]
        dts, nst, pl = [_linear_dt(case, p["kappa"], p["s"]) for p in ps], [case["steps"]] * len(ps), [plans[p["s"]] for p in ps]
        ws = workspace(F.frkc2_batch_workspace_size(pl, probs, nst))
        F.frkc2_batch_prepare(pl, probs, dts, nst, views, ws)
        st.update(plan=pl, prob=probs, u0=u0, flat=flat, views=views, ws=ws)
    else:
        prob = F.make_bruss_problem((case["nx"], case["ny"]), dx=inp["dx"], bc=bc, precision=prec)
        st.update(plan=F.frkc2_plan(case["s"]), prob=prob, dt=_bruss_dt(case, inp["dx"]), v0=inp["v"], w0=inp["w"], v=inp["v"].clone(),
                  w=inp["w"].clone(), ws=workspace(F.frkc2_bruss_workspace_size(prob)))
    return st


def run(state):
    F, kind = state["F"], state["kind"]
    if kind == "adjoint2d":
        u = state["steps_fn"](state["u0"], state["kappa"], state["plan"], state["dt"], state["steps"], bc=state["bc"], precision=state["prec"],
                              ckpt_every=state["ckpt"])
        du, dk = torch.autograd.grad(((u - state["target"]) ** 2).sum(), (state["u0"], state["kappa"]))
        return {"u": u.detach(), "du0": du, "dkappa": dk}
    if kind == "batched2d":
        state["flat"].copy_(state["u0"])
        F.frkc2_batch_launch(state["ws"])
        return state["views"]
    if kind == "bruss2d":
        state["v"].copy_(state["v0"])
        state["w"].copy_(state["w0"])
        F.frkc2_bruss_step(state["plan"], state["prob"], state["dt"], state["steps"], 0.0, state["v"], state["w"], state["ws"])
        return {"v": state["v"], "w": state["w"]}
    state["u"].copy_(state["u0"])
    F.frkc2_step(state["plan"], state["prob"], state["dt"], state["steps"], 0.0, state["u"], state["ws"])
    return state["u"]


def work(case):
    kind, prec = case["kind"], case["prec"]
    sb, kb = (4 if prec == "fp32" else 8), (8 if prec == "fp64" else 4)
    if kind == "batched2d":
        rng = np.random.default_rng(case["count"] * 1000 + case["nmax"])
        sizes = [(int(rng.integers(case["nmin"], case["nmax"] + 1)), int(rng.choice([16, 32, 64, 128]))) for _ in range(case["count"])]
        cells, stages = sum(n * n for n, _ in sizes), sum(n * n * s for n, s in sizes) * case["steps"]
    else:
        cells = case["nx"] * case.get("ny", 1) * case.get("nz", 1)
        stages = cells * case["s"] * case["steps"]
    per_cell = {"heat1d": 2 * sb, "bruss2d": 4 * sb, "adjoint2d": 4 * sb + 2 * kb}.get(kind, 2 * sb + (0 if case.get("kappa") == "power" else kb))
    key = kind + ("_" + case["kappa"] if kind == "step3d" else "")
    return {"bytes": float(cells * per_cell), "flops": float(stages * FLOPS[key])}
