"""Performance cases of the stage solver: what a program that uses it calls,
over the range of sizes, storage kinds and smoothers it is used with.

A case is a dict of plain values.  ``call`` names the entry points:

  assemble   Grid.assemble(u, jacobian=True, F)    F(u), and J and M kept in the grid
  residual   Grid.assemble(u, jacobian=False, F)   F(u) alone
  solve      Grid.solve on an assembled, set-up grid
  stage      Grid.assemble + Grid.gmg_setup + Grid.solve: one stage from scratch
  limex      Grid.limex_step, four columns
  ensemble   limex_step_batched over cubes of the `members` sizes ("33,33,49")
  ie         Grid.ie_step: one implicit Euler step by Newton's method

``nx, ny, nz`` are vertices per axis (nz = 1: 2D).  ``field`` is "lognormal"
(K lognormal with a correlation length of 8 cells and, with `lenses`, boxes of
low K and a higher entry pressure), "lens" (the 33 x 33 square with one lens)
or "layers" (the layered vertical section with an injected light phase).
"""
import math

import numpy as np
import torch

import paper_2506_04763_gb300 as rf
from paper_2506_04763_gb300 import inputs as I

RTOL = 1e-10            # true relative residual of the stage solves (the benchmark's)
H_STAGE = 10.0          # seconds, the stage step of the lognormal workloads
H_DAY = 86400.0         # seconds, the implicit Euler step on the layered section
LIMEX_TOL = 1.0         # loose: the step is accepted and the new state comes back
ENSEMBLE_SIZES = (33, 49, 65, 97)


def _case(name, call, n, field="lognormal", precision="fp32", smoother="gs8", lenses=0, members="", rtol=RTOL):
    c = dict(call=call, nx=n[0], ny=n[1], nz=n[2], field=field, precision=precision, smoother=smoother,
             lenses=lenses, members=members, rtol=rtol)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest problem a user assembles: a 2D test square, launches only
        _case("assemble-2d-33", "assemble", (33, 33, 1), field="lens"),
        # F alone: every substep of a LIMEX column and every line search; the
        # largest grid of the ensemble
        _case("residual-3d-97", "residual", (97, 97, 97)),
        # F, J and M of an ordinary 3D grid with lenses (upwind, cap and clamp branches)
        _case("assemble-3d-129", "assemble", (129, 129, 129), lenses=6),
        # a linear solve of the fixed-step scheme: 2D, all FP64, loose tolerance
        _case("solve-2d-257x129-fp64", "solve", (257, 129, 1), field="layers", precision="fp64", rtol=1e-6),
        # a stage solve of the 65^3 workload: FP64 preconditioner, block Jacobi
        _case("solve-3d-65-fp64", "solve", (65, 65, 65), precision="fp64", smoother="jacobi"),
        # FP16 storage of the finest matrix
        _case("solve-3d-129-fp16", "solve", (129, 129, 129), precision="fp16", lenses=6),
        # the benchmark's solve
        _case("solve-3d-257-fp32", "solve", (257, 257, 257), lenses=6),
        # one stage from scratch on an uneven box (a reservoir section), block Jacobi
        _case("stage-3d-161x97x65", "stage", (161, 97, 65), smoother="jacobi", lenses=6),
        # one stage from scratch at the benchmark's size: the largest case
        _case("stage-3d-257", "stage", (257, 257, 257), lenses=6),
        # one LIMEX step of the 65^3 workload
        _case("limex-3d-65-fp64", "limex", (65, 65, 65), precision="fp64", smoother="jacobi"),
        # a small ensemble: two members of each grid size, one LIMEX step each
        _case("ensemble-8", "ensemble", (0, 0, 0), smoother="jacobi", members="33,33,49,49,65,65,97,97"),
        # one day of the layered section with implicit Euler
        _case("ie-2d-257x129-fp64", "ie", (257, 129, 1), field="layers", precision="fp64", rtol=1e-6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["assemble", "residual", "solve", "stage", "limex", "ensemble", "ie"])
    precision = rng.choice(["fp64", "fp32", "fp16"])
    smoother = rng.choice(["gs8", "jacobi"])
    lenses = rng.choice([0, 6])
    if call in ("assemble", "residual"):
        # any box: assembly needs no hierarchy
        if rng.random() < 0.3:
            n = (_log_int(rng, 9, 900), _log_int(rng, 9, 900), 1)
        else:
            n = (_log_int(rng, 9, 200), _log_int(rng, 9, 200), _log_int(rng, 9, 200))
        return _case(None, call, n, lenses=lenses)
    if call == "ensemble":
        sizes = sorted(rng.choice(ENSEMBLE_SIZES) for _ in range(rng.randint(3, 10)))
        return _case(None, call, (0, 0, 0), smoother="jacobi", members=",".join(map(str, sizes)))
    if call == "ie":
        # sections of about the layered problem's shape, elements 1 to 8 m
        k = rng.choice([3, 4, 5])
        n = ((rng.randint(8, 11) << k) + 1, (rng.randint(3, 5) << k) + 1, 1)
        return _case(None, call, n, field="layers", precision="fp64", smoother="gs8", rtol=1e-6)
    # nested boxes (m 2^k + 1 vertices per axis) down to a coarsest grid of at most 6 cells per axis
    if rng.random() < 0.25:
        k = rng.choice([3, 4, 5, 6])
        n = tuple((rng.randint(2, 6) << k) + 1 for _ in range(2)) + (1,)
    else:
        k = rng.choice([2, 3, 4] if call == "limex" else [2, 3, 4, 5])
        n = tuple((rng.randint(2, 5) << k) + 1 for _ in range(3))
    return _case(None, call, n, precision=precision, smoother=smoother, lenses=lenses)


# ------------------------------------------------------------------ problems
def _levels(n):
    """Vertex-nested levels of a box, down to at most 5 vertices on its longest axis."""
    m = [t for t in n if t > 1]
    L = 1
    while all((t - 1) % 2 == 0 for t in m) and max(m) > 5 and min(m) >= 5:
        m = [(t - 1) // 2 + 1 for t in m]
        L += 1
    return L


def _lognormal(n, seed, lenses):
    """A box with cubic cells, its longest edge 1 m: K, p_d, state and boundary
    data as in the lognormal workloads, drawn on the GPU."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    dim = 3 if n[2] > 1 else 2
    cells = [max(1, t - 1) for t in n]                                 # x, y, z
    h = tuple([1.0 / (max(n) - 1)] * dim + [1.0] * (3 - dim))
    ell, pad = 8.0, 24
    f = torch.randn([c + 2 * pad if c > 1 else 1 for c in cells[::-1]], generator=gen, device=dev, dtype=torch.float64)
    for axis, c in enumerate(cells[::-1]):
        if c == 1:
            continue
        d = torch.arange(c, device=dev).view(-1, 1) + pad - torch.arange(c + 2 * pad, device=dev).view(1, -1)
        w = torch.exp(-0.5 * (d.double() / (ell / 2)) ** 2) * (d.abs() <= 16)
        f = torch.movedim(torch.tensordot(w, f, dims=([1], [axis])), 0, axis)
    lnK = math.log(5e-11) + (f - f.mean()) / f.std()
    K = torch.exp(lnK)
    pd = torch.full_like(K, I.SAND["pd"])
    rng = np.random.default_rng(seed)
    for _ in range(lenses):
        box = []
        for c in cells[::-1]:
            ext = min(int(rng.integers(8, 33)), c)
            start = int(rng.integers(0, c - ext + 1))
            box.append(slice(start, start + ext))
        K[tuple(box)] /= 20.0
        pd[tuple(box)] = I.LENS["pd"]
    nv = n[0] * n[1] * n[2]
    v = torch.arange(nv, device=dev)
    x, y, z = (v % n[0]).double() * h[0], (v // n[0] % n[1]).double() * h[1], (v // (n[0] * n[1])).double() * h[2]
    up, nup = (z, n[2]) if dim == 3 else (y, n[1])
    top = (nup - 1) * h[dim - 1]
    on_top = (v // (n[0] * n[1]) if dim == 3 else v // n[0]) == nup - 1
    pw = I.P_TOP + I.FLUIDS["rho_w"] * I.GRAV * (top - up) + 10.0 * torch.randn(nv, generator=gen, device=dev, dtype=torch.float64)
    pw = torch.where(on_top, torch.full_like(pw, I.P_TOP), pw)
    r2 = (x - 0.5 * (n[0] - 1) * h[0]) ** 2 + (up - top) ** 2
    if dim == 3:
        r2 = r2 + (y - 0.5 * (n[1] - 1) * h[1]) ** 2
    sn = (0.3 * torch.exp(-r2 / 0.05)).clamp(0.0, 0.8)
    host = lambda t: t.reshape(-1).cpu().numpy()  # noqa: E731
    return dict(dim=dim, n=tuple(n), h=h, g=(0.0, 0.0, -I.GRAV) if dim == 3 else (0.0, -I.GRAV, 0.0), K=host(K),
                phi=np.full(K.numel(), I.SAND["phi"]), pd=host(pd), dir=host(on_top.to(torch.uint8)),
                pw_dir=host(torch.where(on_top, pw, torch.zeros_like(pw))), q_in=None,
                u0=torch.stack([pw, sn], 1).reshape(-1), **I.FLUIDS, **I.BROOKS_COREY)


def _problem(case, seed):
    n = (case["nx"], case["ny"], case["nz"])
    if case["field"] == "lens":
        p = I.lens_square_2d()
        p["u0"] = torch.tensor(I.initial_state(2, p["n"], p["h"], seed=seed), device="cuda")
        return p
    if case["field"] == "layers":
        # early injection: a thin plume around the injection point, drawn
        p = I.case4_analogue(n[:2])
        rng = np.random.default_rng(seed)
        v = np.arange(n[0] * n[1])
        x, y = (v % n[0]) * p["h"][0], (v // n[0]) * p["h"][1]
        cx, r = 250.0 + rng.uniform(-20.0, 20.0), rng.uniform(25.0, 35.0)
        u = p["u0"].copy()
        u[1::2] += rng.uniform(0.005, 0.02) * np.exp(-(((x - cx) / (2 * r)) ** 2 + ((y - 25.0) / r) ** 2))
        p["u0"] = torch.tensor(u, device="cuda")
        return p
    return _lognormal(n, seed, case["lenses"])


def _members(case):
    """Vertices per axis of each member of an ensemble."""
    return [int(t) for t in case["members"].split(",")]


def _opts(case, n):
    L = I.levels_for(min(n[:2])) if case["field"] == "layers" else _levels(n)
    return rf.gmg_opts(L, case["smoother"], precision=case["precision"])


def prepare(case, seed):
    """The grids and states a program has in hand; for a solve, also the
    assembled operator, its hierarchy and the right-hand side."""
    if case["call"] == "ensemble":
        sizes = _members(case)
        probs = [_lognormal((s, s, s), 1000 * seed + k, 0) for k, s in enumerate(sizes)]
        return dict(case=case, grids=[rf.Grid(p) for p in probs], u0=[p["u0"] for p in probs],
                    u=[p["u0"].clone() for p in probs], gmg=[_opts(case, (s, s, s)) for s in sizes])
    p = _problem(case, seed)
    st = dict(case=case, grid=rf.Grid(p), u0=p["u0"], u=p["u0"].clone(), F=torch.empty_like(p["u0"]),
              x=torch.empty_like(p["u0"]), gmg=_opts(case, p["n"]))
    if case["call"] == "solve":
        st["grid"].assemble(st["u0"], jacobian=True, F=st["F"])
        st["grid"].gmg_setup([1.0 / _step(case)], st["gmg"])
    return st


def _step(case):
    return H_DAY if case["field"] == "layers" else H_STAGE


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "ensemble":
        for u, u0 in zip(state["u"], state["u0"]):
            u.copy_(u0)
        rf.limex_step_batched(state["grids"], state["u"], H_STAGE, kappa=4, tol=LIMEX_TOL, gmg=state["gmg"],
                              rtol=case["rtol"])
        return state["u"]
    g = state["grid"]
    if call in ("assemble", "residual"):
        g.assemble(state["u0"], jacobian=call == "assemble", F=state["F"])
        return state["F"]
    if call == "solve":
        g.solve(0, state["F"], state["x"], rtol=case["rtol"])
        return state["x"]
    if call == "stage":
        g.assemble(state["u0"], jacobian=True, F=state["F"])
        g.gmg_setup([1.0 / _step(case)], state["gmg"])
        g.solve(0, state["F"], state["x"], rtol=case["rtol"])
        return {"F": state["F"], "x": state["x"]}
    state["u"].copy_(state["u0"])
    if call == "limex":
        info = g.limex_step(state["u"], H_STAGE, kappa=4, tol=LIMEX_TOL, gmg=state["gmg"], rtol=case["rtol"])
        return {"u": state["u"], "accepted": info["accepted"]}
    info = g.ie_step(state["u"], H_DAY, atol=1e-8, rtol=1e-6, max_newton=50, gmg=state["gmg"], lin_rtol=case["rtol"])
    return {"u": state["u"], "status": info["status"]}


def work(case):
    """Bytes and operations no implementation avoids, in FP64: states and cell
    data read once, results written once; the Jacobian written once where the
    call leaves it in the grid and read once per linear solve."""
    if case["call"] == "ensemble":
        one = [work(_case(None, "limex", (s, s, s))) for s in _members(case)]
        return {k: sum(w[k] for w in one) for k in ("bytes", "flops")}
    n = (case["nx"], case["ny"], case["nz"])
    nv = n[0] * n[1] * n[2]
    nb, dim = (27, 3) if n[2] > 1 else (9, 2)
    faces = dim << (dim - 1)                      # sub-control-volume faces per element
    resid = {"bytes": nv * (16 + 24 + 16), "flops": nv * faces * 40}
    jac = {"bytes": nv * (32 * nb + 16), "flops": nv * faces * 2 ** dim * 8}
    lin = {"bytes": nv * (32 * nb + 32), "flops": nv * 8 * nb}
    times = dict(assemble=(1, 1, 0), residual=(1, 0, 0), solve=(0, 0, 1), stage=(1, 1, 1), limex=(7, 1, 10),
                 ie=(2, 1, 1))[case["call"]]
    return {k: times[0] * resid[k] + times[1] * jac[k] + times[2] * lin[k] for k in ("bytes", "flops")}


# ------------------------------------------------------------------ 64-bit reference
def _residual_torch(p, u):
    """F(u) of the vertex-centred finite-volume scheme in plain torch (lambda =
    2): per element and axis, the face fluxes between its corner pairs."""
    dev = u.device
    n, h, dim = p["n"], p["h"], p["dim"]
    cz = n[2] - 1 if dim == 3 else 1
    cell = lambda k: torch.as_tensor(p[k], device=dev).reshape(cz, n[1] - 1, n[0] - 1)  # noqa: E731
    K, pd = cell("K"), cell("pd")
    pw, sn = u.reshape(n[2], n[1], n[0], 2).unbind(-1)
    den = 1.0 - p["S_wr"] - p["S_nr"]
    se = (1.0 - sn - p["S_wr"]) / den

    def corner(a, q):                             # the elements' corner q of a vertex field
        sl = [slice(q >> t & 1, a.shape[2 - t] - 1 + (q >> t & 1)) if t < dim else slice(None) for t in range(3)]
        return a[sl[2], sl[1], sl[0]]

    pdm = torch.full_like(pw, math.inf)
    for q in range(1 << dim):
        view = corner(pdm, q)
        view.copy_(torch.minimum(view, pd))
    lev = torch.where(se < 0.01, 10.0 - 500.0 * (se - 0.01),
                      torch.where(se > 1.0, 1.0 - 0.5 * (se - 1.0), se.clamp(min=0.01) ** -0.5))
    pc = pdm * lev
    pn = pw + pc
    krw = lambda s: s.clamp(0.0, 1.0) ** 4  # noqa: E731
    Fw, Fn = torch.zeros_like(pw), torch.zeros_like(pw)
    for k in range(dim):
        oth = [t for t in range(dim) if t != k]
        KA = K * math.prod(h[t] / 2 for t in oth)
        dn, dc, av = {}, {}, {}
        for a in (q for q in range(1 << dim) if not q >> k & 1):
            b = a | 1 << k
            dn[a], dc[a] = corner(pn, b) - corner(pn, a), corner(pc, b) - corner(pc, a)
            av[a] = 0.5 * (corner(se, a) + corner(se, b))
        for a in dn:
            b = a | 1 << k
            w = {a2: math.prod(0.75 if (a2 ^ a) >> t & 1 == 0 else 0.25 for t in oth) for a2 in dn}
            gn, gc, sM = (sum(w[a2] * v[a2] for a2 in dn) for v in (dn, dc, av))
            Tw = -KA * (gn / h[k] - p["rho_w"] * p["g"][k])
            Tn = -KA * (gn / h[k] - p["rho_n"] * p["g"][k])
            Tc = -KA * (gc / h[k])
            up = Tw >= 0
            lw = krw(torch.where(up, corner(se, a), corner(se, b))) / p["mu_w"]
            up = Tn >= 0
            s, m = torch.where(up, corner(se, a), corner(se, b)), torch.where(up, corner(pdm, a), corner(pdm, b))
            s = torch.where(pd == m, s, ((pd / m) ** 2 * s).clamp(max=1.0)).clamp(0.0, 1.0)
            fw = p["rho_w"] * (lw * Tw - krw(sM) / p["mu_w"] * Tc)
            fn = p["rho_n"] * (((1 - s) ** 2 * (1 - s * s)) / p["mu_n"] * Tn)
            for f, out in ((fw, Fw), (fn, Fn)):
                corner(out, a).sub_(f)
                corner(out, b).add_(f)
    F = torch.stack([Fw, Fn], -1).reshape(-1, 2)
    if p["q_in"] is not None:
        F += torch.as_tensor(p["q_in"], device=dev).reshape(-1, 2)
    fixed = torch.as_tensor(p["dir"], device=dev).bool()
    F[:, 0] = torch.where(fixed, torch.as_tensor(p["pw_dir"], device=dev) - pw.reshape(-1), F[:, 0])
    return F.reshape(-1)


def exact(case, seed):
    """F of the assembling calls.  The linear solves and steps stop at their
    tolerances, and solving these systems exactly without a multigrid method
    takes too long: they have no such value."""
    if case["call"] not in ("assemble", "residual", "stage"):
        return None
    p = _problem(case, seed)
    F = _residual_torch(p, p["u0"])
    return {"F": F, "x": None} if case["call"] == "stage" else F
