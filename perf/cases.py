"""The calls whose speed counts: residuals and RK4 steps of the flow solver, the batched poll with its wall forces
and surface records, and the FW-H integration with the Welch spectrum, at the sizes of this repository's workloads.

``listed`` and ``draw`` give cases (plain dicts), ``prepare`` what a program holds before the call, ``run`` one pass
through the public entry points, ``work`` what the pass cannot do without, ``exact`` the same outputs in 64 bits from
plain torch (Flux Reconstruction, sampling, forces, FW-H and Welch written out here from their definitions).
"""
import math

import numpy as np
import torch

from paper_2501_05709_gb300 import cases as C
from paper_2501_05709_gb300 import fr as F
from paper_2501_05709_gb300 import workloads as W

GAMMA, PRANDTL = 1.4, 0.71
MONO_T0 = 0.25   # time of the monopole runs' first step
PREC = {"fp64": F.FR_FP64, "fp32": F.FR_FP32}


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the 2D isentropic-vortex box (16 x 16, p = 2, Euler, FP64): the smallest call, latency and launches
        {"name": "vortex2d_p2_fp64", "kind": "residual", "mesh": "vortex", "n": 16, "p": 2, "prec": "fp64"},
        # one residual of a curved Navier-Stokes box of odd sizes at p = 2: a caller's own integrator
        {"name": "curved_p2_fp32", "kind": "residual", "mesh": "curved", "nx": 23, "ny": 17, "nz": 13, "p": 2, "prec": "fp32"},
        # one FP64 residual of the coarse airfoil O-grid of the precision study
        {"name": "ogrid_p3_fp64", "kind": "residual", "mesh": "ogrid", "nx": 60, "ny": 20, "nz": 2, "first": 2e-2, "p": 3,
         "prec": "fp64"},
        # the headline workload: Taylor-Green box of 32^3 hexes, p = 3, RK4 steps replayed from the graph
        {"name": "tgv32_p3_fp32", "kind": "step", "mesh": "tgv", "n": 32, "p": 3, "prec": "fp32", "steps": 4},
        # the same box at p = 4
        {"name": "tgv32_p4_fp32", "kind": "step", "mesh": "tgv", "n": 32, "p": 4, "prec": "fp32", "steps": 2},
        # the double-precision solver on a smaller box: what every FP32 result is checked against
        {"name": "tgv16_p3_fp64", "kind": "step", "mesh": "tgv", "n": 16, "p": 3, "prec": "fp64", "steps": 2},
        # one airfoil candidate at full size: 100,000 curved hexes, walls and far field
        {"name": "ogrid100k_p3_fp32", "kind": "step", "mesh": "ogrid", "nx": 250, "ny": 100, "nz": 4, "first": 2e-3, "p": 3,
         "prec": "fp32", "steps": 2},
        # an airfoil candidate with the far-field sponge of lower degrees
        {"name": "sponge_p3_fp32", "kind": "step", "mesh": "ogrid", "nx": 125, "ny": 50, "nz": 4, "first": 5e-3, "p": 3,
         "prec": "fp32", "steps": 4, "sponge": True},
        # the monopole box of 125,000 hexes: Euler, far field, energy source, adaptive time step
        {"name": "monopole50_p2_fp32", "kind": "step", "mesh": "monopole", "n": 50, "p": 2, "prec": "fp32",
         "steps": 4, "cfl": 0.5},
        # a poll of the design loop: uneven candidates in one context, wall forces, surface records every 4th step
        {"name": "poll12_p3_fp32", "kind": "poll", "cands": 12, "lo": 30, "hi": 56, "nz": 2, "first": 2e-2, "p": 3,
         "prec": "fp32", "steps": 40, "every": 4},
        # one observer of one candidate and its spectrum: the objective of the design loop
        {"name": "fwh_observer", "kind": "fwh", "spacing": 0.05, "obs": 1, "copies": 1, "nt": 2400, "nseg": 3},
        # the directivity circle: 18,840 panels, 36 observers, three span copies, and the spectra
        {"name": "fwh_directivity", "kind": "fwh", "spacing": 0.01, "obs": 36, "copies": 3, "nt": 1000, "nseg": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vortex", "curved", "ogrid_res", "tgv", "tgv", "tgv64", "ogrid", "sponge", "monopole", "poll",
                       "fwh", "fwh"])
    if kind == "vortex":
        return {"kind": "residual", "mesh": "vortex", "n": _log(rng, 12, 96), "p": rng.randint(1, 4),
                "prec": rng.choice(["fp64", "fp32"])}
    if kind == "curved":
        return {"kind": "residual", "mesh": "curved", "nx": _log(rng, 5, 28), "ny": _log(rng, 5, 28),
                "nz": _log(rng, 5, 28), "p": rng.randint(1, 4),
                "prec": rng.choice(["fp64", "fp32"])}
    if kind == "ogrid_res":
        return {"kind": "residual", "mesh": "ogrid", "nx": _log(rng, 30, 90), "ny": _log(rng, 10, 30),
                "nz": rng.randint(1, 3), "first": 2e-2, "p": rng.randint(2, 3), "prec": "fp64"}
    if kind == "tgv":
        return {"kind": "step", "mesh": "tgv", "n": _log(rng, 7, 32), "p": rng.randint(2, 4), "prec": "fp32",
                "steps": rng.randint(1, 4)}
    if kind == "tgv64":
        return {"kind": "step", "mesh": "tgv", "n": _log(rng, 5, 20), "p": rng.randint(2, 4), "prec": "fp64",
                "steps": rng.randint(1, 2)}
    if kind in ("ogrid", "sponge"):
        return {"kind": "step", "mesh": "ogrid", "nx": _log(rng, 40, 200), "ny": _log(rng, 20, 80),
                "nz": rng.randint(2, 4), "first": 5e-3, "p": rng.randint(3, 4) if kind == "ogrid" else 3, "prec": "fp32",
                "steps": rng.randint(1, 3), "sponge": kind == "sponge"}
    if kind == "monopole":
        return {"kind": "step", "mesh": "monopole", "n": _log(rng, 15, 50), "p": rng.randint(1, 3), "prec": "fp32",
                "steps": rng.randint(1, 4), "cfl": rng.choice([0.0, 0.5])}
    if kind == "poll":
        return {"kind": "poll", "cands": rng.randint(3, 12), "lo": rng.randint(26, 40), "hi": rng.randint(44, 60),
                "nz": 2, "first": 2e-2, "p": 3, "prec": "fp32", "steps": rng.randint(8, 40), "every": rng.randint(1, 8)}
    return {"kind": "fwh", "spacing": round(math.exp(rng.uniform(math.log(0.016), math.log(0.1))), 4),
            "obs": _log(rng, 1, 36), "copies": rng.choice([1, 3]), "nt": _log(rng, 900, 2400), "nseg": 3}


# ---------------------------------------------------------------- inputs
def _gl(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x - x[::-1]), 0.5 * (w + w[::-1])


def _lagr(xs, ys):
    return np.array([[np.prod([(y - xs[m]) / (xs[j] - xs[m]) for m in range(len(xs)) if m != j])
                      for j in range(len(xs))] for y in ys])


def _dlagr(xs, ys):
    n = len(xs)
    return np.array([[sum(np.prod([(y - xs[m]) / (xs[j] - xs[m]) for m in range(n) if m not in (j, k)])
                          / (xs[j] - xs[k]) for k in range(n) if k != j) for j in range(n)] for y in ys], dtype=float)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _along(a, M, d):
    """a [..., n_{dim-1}, .., n_0] with the matrix M [m, n] applied along direction d (n_0 is direction 0)."""
    ax = a.ndim - 1 - d
    return torch.tensordot(a, M, dims=([ax], [1])).movedim(-1, ax)


def _points(nodes, p):
    """Physical solution points [E, nsp, dim] of an element map through equispaced nodes."""
    E, nn, dim = nodes.shape
    q = int(round(nn ** (1.0 / dim)))
    X = _dev(nodes).movedim(-1, 1).reshape((E, dim) + (q,) * dim)
    B = _dev(_lagr(np.linspace(-1, 1, q), _gl(p + 1)[0]))
    for d in range(dim):
        X = _along(X, B, d)
    return X.reshape(E, dim, -1).movedim(1, -1)


def _conserved(rho, V, pr):
    """[E, nv, nsp] from rho, pr [E, nsp] and V, a list of [E, nsp]."""
    ke = 0.5 * rho * sum(v * v for v in V)
    return torch.stack([rho] + [rho * v for v in V] + [pr / (GAMMA - 1.0) + ke], dim=1)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _shape(case):
    return [case["nx"], case["ny"], case["nz"]]


def _sizes(case):
    """(n_theta, n_r) of each candidate of a poll: uneven, from lo to hi around the section."""
    k, a, b = case["cands"], case["lo"], case["hi"]
    nt = [a + (b - a) * i // max(1, k - 1) for i in range(k)]
    return [(n, 2 * n // 5) for n in nt]


def _flow(case, seed):
    """Meshes, options, per-candidate steps and the initial state of a flow case (values that FP32 holds exactly
    when the solver works in FP32)."""
    p, prec, mesh = case["p"], PREC[case["prec"]], case.get("mesh", "poll")
    g = _gen(seed)
    rnd = lambda shape: 2.0 * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 1.0
    ph = [float(v) for v in rnd((8,)).cpu()]
    dts, caps = None, None
    if mesh == "vortex":
        # the vortex with a phase and an amplitude of its own
        n = case["n"]
        meshes = [W.box_mesh(2, n, -5.0, 5.0, q=1)]
        opts = F.options(order=p, precision=prec, vel_inf=(0.5 * math.sqrt(GAMMA), 0.0, 0.0))
        x = _points(meshes[0][0], p)
        dx, dy = x[..., 0] - 0.5 * ph[0], x[..., 1] - 0.5 * ph[1]
        b = 5.0 + 0.5 * ph[2]
        r2 = dx * dx + dy * dy
        f = b / (2 * math.pi) * torch.exp(0.5 * (1.0 - r2))
        T = 1.0 - (GAMMA - 1.0) * b * b / (8.0 * GAMMA * math.pi ** 2) * torch.exp(1.0 - r2)
        rho = T ** (1.0 / (GAMMA - 1.0))
        u = _conserved(rho, [0.5 * math.sqrt(GAMMA) - dy * f, dx * f], rho ** GAMMA)
    elif mesh == "curved":
        # a smooth O(1) flow on a curved periodic box, at least four elements to a wave, at the airfoil's Reynolds number
        meshes = [W.box_mesh(3, _shape(case), 0.0, 1.0, q=2, curve=0.1, seed=2)]
        opts = F.options(order=p, precision=prec, viscous=True, mu=1.0 / 23000.0)
        x = 2 * math.pi * _points(meshes[0][0], p) * _dev(np.maximum(1, np.array(_shape(case)) // 4))
        s = lambda k, c: torch.sin(x[..., k % 3] + math.pi * c) * torch.cos(x[..., (k + 1) % 3])
        u = _conserved(1.0 + 0.2 * s(0, ph[0]), [0.3 + 0.2 * s(k, ph[k]) for k in (1, 2, 3)], 1.0 + 0.2 * s(4, ph[4]))
    elif mesh == "tgv":
        # Taylor-Green vortex at Mach 0.1 plus 1% of seeded velocity noise
        meshes = [W.box_mesh(3, case["n"], 0.0, 2 * math.pi, q=1)]
        p0 = 1.0 / (GAMMA * 0.01)
        opts = F.options(order=p, precision=prec, viscous=True, mu=1.0 / 1600.0, p_inf=p0,
                         dt=(2.5e-4 if p <= 3 else 1.5e-4))
        X, Y, Z = _points(meshes[0][0], p).unbind(-1)
        pr = p0 + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
        V = [torch.sin(X) * torch.cos(Y) * torch.cos(Z), -torch.cos(X) * torch.sin(Y) * torch.cos(Z), torch.zeros_like(X)]
        u = _conserved(pr / p0, [v + 0.01 * rnd(X.shape) for v in V], pr)
    elif mesh == "monopole":
        # the quiescent box with weak seeded noise
        nodes, conn, opts, _ = C.monopole_box_setup(case["n"], p, prec)
        meshes = [(nodes, conn)]
        E, nsp = len(nodes), (p + 1) ** 3
        one = torch.ones((E, nsp), device="cuda", dtype=torch.float64)
        u = _conserved(one, [1e-3 * rnd((E, nsp)) for _ in range(3)], one / GAMMA)
    else:
        # airfoil O-grids in the perturbed free stream at 3 degrees, each candidate at its stable step
        if mesh == "ogrid":
            shapes = [(_shape(case), (0.02, 0.4, 0.12))]
        else:
            shapes = [([a, b, case["nz"]], (0.01 * (k % 6), 0.3 + 0.02 * k, 0.1 + 0.005 * k))
                      for k, (a, b) in enumerate(_sizes(case))]
        meshes, dts = [], []
        for (nt, nr, nz), naca in shapes:
            nodes, conn, opts, (rho, vel, pr) = C.naca_setup(naca, nt, nr, nz, first_cell=case["first"], order=p,
                                                             precision=prec)
            meshes.append((nodes, conn))
            dts.append(C.stable_dt(nodes, nt, order=p))
        opts.dt = dts[0]
        one = torch.ones((sum(len(m[0]) for m in meshes), (p + 1) ** 3), device="cuda", dtype=torch.float64)
        u = _conserved(rho * one, [float(vel[i]) + 0.01 * rnd(one.shape) for i in range(3)], pr * one)
        if case.get("sponge"):
            caps = W.sponge_orders(meshes[0][0], p)
    u = u.contiguous()
    if case["prec"] == "fp32":
        u = u.float().double()
    return meshes, opts, dts, u, caps


RING = [(-0.5, 0.1, -0.5), (0.5, 0.1, -0.5), (-0.5, 0.1, 0.5), (0.5, 0.1, 0.5)]  # reference places of surface points


def _surface(nodes, nt, nr, nz):
    """Elements and points of a data surface: the O-grid ring nearest to 1.5 chords from mid-chord."""
    mid = nodes[:nt * nr].mean(axis=1)
    rad = np.hypot(mid[:, 0] - 0.5, mid[:, 1]).reshape(nr, nt).mean(axis=1)
    i = int(np.argmin(np.abs(rad - 1.5)))
    el = np.concatenate([np.arange(nt) + nt * (i + nr * k) for k in range(nz)])
    q = 3
    B = [_lagr(np.linspace(-1, 1, q), [xi[d] for xi in RING]) for d in range(3)]
    w = np.einsum("kc,kb,ka->kcba", B[2], B[1], B[0]).reshape(len(RING), -1)
    return el, np.ascontiguousarray(np.einsum("kn,eni->eki", w, nodes[el]).reshape(-1, 3))


def _fwh_inputs(case, seed):
    """A seeded record on a closed cylinder of 1.5 chords: sound of four sources inside it and a convected
    disturbance, in the moving medium of the airfoil workloads (|V| = 1, M = 0.2, 3 degrees)."""
    y, n, dS = W.cylinder_surface(radius=1.5, center=(0.5, 0.0), spacing=case["spacing"], span=0.2)
    nt, c0, a = case["nt"], 5.0, math.radians(3.0)
    dt = 0.002 * max(1.0, 1000.0 / nt) if case["obs"] > 1 else 1.6e-3
    M = [0.2 * math.cos(a), 0.2 * math.sin(a), 0.0]
    p0 = c0 * c0 / GAMMA
    yd, nd, sd = _dev(y), _dev(n), _dev(dS)
    t = dt * torch.arange(nt, device="cuda", dtype=torch.float64)[:, None]
    r = torch.rand((4, 4), generator=_gen(seed), device="cuda", dtype=torch.float64).cpu().numpy()
    U = [c0 * m for m in M]
    pp = torch.zeros((nt, len(y)), device="cuda", dtype=torch.float64)
    vel = [torch.full_like(pp, U[i]) for i in range(3)]
    for amp, om, at, phase in r:
        src = torch.tensor([at, 0.05 * (phase - 0.5), 0.1], device="cuda", dtype=torch.float64)
        d = yd - src
        R = d.norm(dim=1)
        w = 1e-3 * (0.5 + amp) / R * torch.sin(4 * math.pi * (0.5 + om) * (t - R / c0) + 6.28 * phase)
        pp += w
        for i in range(3):
            vel[i] += w / c0 * d[:, i] / R
    vel[1] += 5e-3 * torch.sin(2 * math.pi * (3.0 + r[0, 0]) * (t - yd[:, 0]) + 6.28 * r[0, 1])
    hist = torch.stack([1.0 + pp / (c0 * c0)] + vel + [p0 + pp], dim=-1).contiguous()
    ang = np.radians(np.arange(case["obs"]) * 360.0 / case["obs"] - 90.0)
    obs = np.stack([0.5 + 10.0 * np.cos(ang), 10.0 * np.sin(ang), np.full_like(ang, 0.1)], axis=1)
    return {"hist": hist, "y": yd, "n": nd, "dS": sd, "dt": dt, "obs": obs, "M": M, "c0": c0, "p0": p0}


# ---------------------------------------------------------------- prepare and run
class State:
    """A context and the buffers of its calls; closes the context when it goes."""
    ctx = None

    def __del__(self):
        if self.ctx is not None:
            self.ctx.close()


def prepare(case, seed):
    s = State()
    s.case = case
    if case["kind"] == "fwh":
        s.rec = _fwh_inputs(case, seed)
        return s
    meshes, opts, dts, u, caps = _flow(case, seed)
    s.ctx = F.fr_mesh_load(meshes, opts)
    if case["kind"] == "residual":
        s.u = u.to(torch.float64 if case["prec"] == "fp64" else torch.float32)
        s.R = torch.empty_like(s.u)
        return s
    s.u, s.out = u, torch.empty_like(u)
    if caps is not None:
        F.fr_set_element_order(s.ctx, caps)
    if case.get("mesh") == "monopole":
        F.fr_set_source(s.ctx, 0, C.MONOPOLE_SOURCE, MONO_T0)
        if case["cfl"] > 0.0:
            F.fr_set_adaptive_dt(s.ctx, case["cfl"])
    if case["kind"] == "poll":
        s.surf = []
        for k, (nt, nr) in enumerate(_sizes(case)):
            F.fr_set_cand_dt(s.ctx, k, dts[k])
            pts = _surface(meshes[k][0], nt, nr, case["nz"])[1]
            cap = (case["steps"] + case["every"] - 1) // case["every"]
            s.surf.append((F.fwh_register(s.ctx, k, pts, cap, case["every"]), len(pts)))
    return s


def run(s):
    case, st = s.case, torch.cuda.current_stream().cuda_stream
    if case["kind"] == "residual":
        F.fr_residual(s.ctx, s.u, s.R, stream=st)
        return {"R": s.R}
    if case["kind"] == "fwh":
        r = s.rec
        p, nt, t0 = F.fwh_integrate(r["hist"], r["y"], r["n"], r["dS"], r["dt"], 0.0, r["obs"], r["M"], r["c0"], 1.0,
                                    r["p0"], Lspan=0.2, ncopies=case["copies"], stream=st)
        psd, freq = F.fwh_psd(p, r["dt"], nseg=case["nseg"], nt=int(nt.min()), stream=st)
        return {"p": p, "nt": nt, "t0": t0, "psd": psd, "freq": freq}
    # a run from its initial state: device state in, graph-replayed steps, device state out
    if case["kind"] == "poll":
        F.fr_forces_reset(s.ctx)
        for h, _ in s.surf:
            F.fwh_clear(s.ctx, h)
    F.fr_state_set(s.ctx, s.u, stream=st)
    F.fr_rk_step_graph(s.ctx, case["steps"], stream=st)
    F.fr_state_get(s.ctx, out=s.out, stream=st)
    got = {"u": s.out}
    if case["kind"] == "poll":
        got["forces"] = np.stack([F.fr_forces(s.ctx, k) for k in range(s.ctx.ncand)])
        got["records"] = [F.fwh_history(s.ctx, h, n) for h, n in s.surf]
    return got


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    if case["kind"] == "fwh":
        npts = int(round(3 * math.pi / case["spacing"])) * int(round(0.2 / case["spacing"]))
        pcos = npts * case["copies"] * case["obs"] * case["nt"]
        # eight source series combined and four stencil weights per panel, copy, observer and sample
        return {"bytes": 8.0 * (5 * npts * case["nt"] + 2 * case["obs"] * case["nt"]), "flops": 24.0 * pcos}
    p = case["p"]
    if case["kind"] == "poll":
        E, dim, curved = sum(a * b for a, b in _sizes(case)) * case["nz"], 3, True
    elif case["mesh"] == "vortex":
        E, dim, curved = case["n"] ** 2, 2, False
    else:
        curved = case["mesh"] in ("curved", "ogrid")
        E, dim = (int(np.prod(_shape(case))) if curved else case["n"] ** 3), 3
    visc = case.get("mesh") not in ("vortex", "monopole")
    rsz = 8 if case["prec"] == "fp64" else 4
    n, nv = p + 1, dim + 2
    nsp, nfp = n ** dim, n ** (dim - 1)
    sz = rsz if case["kind"] == "residual" else 8
    geo = (dim * dim + 1) * nsp + 2 * dim * nfp * dim if curved else dim * dim + 1 + 2 * dim * dim
    lines = dim * nv * nfp
    # per evaluation: traces, (corrected gradient, face gradient,) divergence and correction; point-wise fluxes
    fl = lines * (4 * n + 2 * n * n + 8 * n) + nsp * 60 + 2 * dim * nfp * 70
    if visc:
        fl += lines * (2 * n * n + 4 * n) + 2 * dim * nfp * (2 * n * nv * dim + 90) + nsp * (100 + (90 if curved else 20))
    evals = 1 if case["kind"] == "residual" else 4 * case["steps"]
    return {"bytes": float(E * (2 * nv * nsp * sz + geo * rsz)), "flops": float(E * fl * evals)}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
class _Ref:
    """1D operators of degree q (DG correction)."""

    def __init__(self, q):
        self.x, self.w = _gl(q + 1)
        P = np.polynomial.legendre.Legendre
        c = np.zeros(q + 2)
        c[q + 1], c[q] = 1.0, -1.0
        g = P(0.5 * (-1.0) ** (q + 1) * c).deriv()       # derivative of the right Radau polynomial
        self.lm, self.lp = _dev(_lagr(self.x, [-1.0])[0]), _dev(_lagr(self.x, [1.0])[0])
        self.D = _dev(_dlagr(self.x, self.x))
        self.hm, self.hp = _dev(-g(self.x)), _dev(-g(-self.x))
        inner = np.sort(np.real(P.basis(q).deriv().roots())) if q > 1 else np.zeros(0)
        self.gll = np.concatenate([[-1.0], inner, [1.0]])


def _end(a, v, d):
    return torch.tensordot(a, v, dims=([a.ndim - 1 - d], [0]))


def _spread(fv, h, d, dim, n):
    """Face values [..., n^(dim-1)] along the lines normal to the face, with the profile h."""
    return fv.reshape(fv.shape[:-1] + (n,) * (dim - 1)).unsqueeze(-1 - d) * h.reshape((n,) + (1,) * d)


class _Geom:
    def __init__(self, nodes, conn, p):
        E, nn, dim = nodes.shape
        self.E, self.dim, self.p = E, dim, p
        self.ref = ref = _Ref(p)
        q = int(round(nn ** (1.0 / dim)))
        xe = np.linspace(-1, 1, q)
        X = _dev(nodes)
        X = (X - X.mean(dim=1, keepdim=True)).movedim(-1, 1).reshape((E, dim) + (q,) * dim)

        def tens(f, mats):
            for d in range(dim):
                f = _along(f, _dev(mats[d]), d)
            return f
        gp = lambda pts, dk: tens(X, [(_dlagr if d == dk else _lagr)(xe, pts) for d in range(dim)])
        A = torch.stack([gp(ref.x, k).reshape(E, dim, -1) for k in range(dim)], dim=2)
        if dim == 2:
            self.J = A[:, 0, 0] * A[:, 1, 1] - A[:, 0, 1] * A[:, 1, 0]
        else:
            a, b, c = A[:, :, 0], A[:, :, 1], A[:, :, 2]
            self.J = (a * torch.linalg.cross(b, c, dim=1)).sum(1)
        xg = gp(ref.gll, -1)
        ag = [gp(ref.gll, k) for k in range(dim)]

        def smetric(pts):
            I, Dm = [_lagr(ref.gll, s) for s in pts], [_dlagr(ref.gll, s) for s in pts]
            ev = lambda f, dk: tens(f, [Dm[d] if d == dk else I[d] for d in range(dim)]).reshape(E, -1)
            if dim == 2:
                x, y = xg[:, 0], xg[:, 1]
                return torch.stack([torch.stack([ev(y, 1), -ev(x, 1)], 1), torch.stack([-ev(y, 0), ev(x, 0)], 1)], 1)
            rows = [[None] * 3 for _ in range(3)]
            for n in range(3):
                l, m = (n + 1) % 3, (n + 2) % 3
                w = [xg[:, l] * ag[k][:, m] for k in range(3)]
                for d in range(3):
                    d1, d2 = (d + 1) % 3, (d + 2) % 3
                    rows[d][n] = ev(w[d2], d1) - ev(w[d1], d2)
            return torch.stack([torch.stack(r, 1) for r in rows], 1)
        self.S = smetric([ref.x] * dim)                                   # [E, d, i, nsp]
        nfp = (p + 1) ** (dim - 1)
        N = torch.empty((E, 2 * dim, dim, nfp), device="cuda", dtype=torch.float64)
        for f in range(2 * dim):
            pts = [ref.x] * dim
            pts[f // 2] = np.array([1.0 if f % 2 else -1.0])
            N[:, f] = (1.0 if f % 2 else -1.0) * smetric(pts)[:, f // 2]
        cn = _dev(conn.astype(np.int64))
        self.tag = torch.where(cn[..., 0] < 0, -cn[..., 0], torch.zeros_like(cn[..., 0]))
        me = torch.arange(E * 2 * dim, device="cuda").reshape(E, 2 * dim)
        self.nb = torch.where(self.tag > 0, me, cn[..., 0] * 2 * dim + cn[..., 1])
        flat = N.reshape(E * 2 * dim, dim, nfp)
        self.N = torch.where((me > self.nb)[..., None, None], -flat[self.nb.reshape(-1)].reshape(N.shape), N)


def _press(u):
    return (GAMMA - 1.0) * (u[:, -1] - 0.5 * (u[:, 1:-1] ** 2).sum(1) / u[:, 0])


def _fluxes(u, G, mu, dim):
    """[K, nv, dim, ...]: inviscid minus viscous flux (G: gradients [K, nv, dim, ...] or None)."""
    V, pr = u[:, 1:-1] / u[:, :1], _press(u)
    Fi = u[:, :, None] * V[:, None]
    for i in range(dim):
        Fi[:, 1 + i, i] += pr
        Fi[:, -1, i] += pr * V[:, i]
    return Fi if G is None else Fi - _visc(u, G, mu, dim)


def _visc(u, G, mu, dim):
    rho, V = u[:, :1], u[:, 1:-1] / u[:, :1]
    gV = (G[:, 1:-1] - V[:, :, None] * G[:, :1]) / rho[:, :, None]
    gE = (G[:, -1] - (u[:, -1:] / rho) * G[:, 0]) / rho
    ge = gE - (V[:, :, None] * gV).sum(1)
    tau = mu * (gV + gV.transpose(1, 2))
    div = sum(gV[:, i, i] for i in range(dim))
    for i in range(dim):
        tau[:, i, i] -= (2.0 / 3.0) * mu * div
    out = torch.zeros_like(G)
    out[:, 1:-1] = tau
    out[:, -1] = (V[:, :, None] * tau).sum(1) + mu * GAMMA / PRANDTL * ge
    return out


class _Solver:
    def __init__(self, geom, opts, caps=None):
        self.g, self.o, self.dim = geom, opts, geom.dim
        self.visc, self.mu = bool(opts.viscous), float(opts.mu)
        dim, p = geom.dim, geom.p
        xp, wp = _gl(p + 1)
        self.groups = []
        leg = lambda k, x: np.polynomial.legendre.Legendre.basis(k)(x)
        for q in range(p + 1):
            sel = None if caps is None else _dev(np.nonzero(np.asarray(caps) == q)[0])
            if (caps is None and q < p) or (sel is not None and len(sel) == 0):
                continue
            r = _Ref(q)
            Iqp, Ipq = _dev(_lagr(xp, r.x)), _dev(_lagr(r.x, xp))
            Pqp = _dev(sum(np.outer(leg(k, r.x), leg(k, xp) * wp) * (2 * k + 1) / 2 for k in range(q + 1)))
            S, J = (geom.S, geom.J) if sel is None else (geom.S[sel], geom.J[sel])
            if q < p:
                S, J = self.vol(S, Iqp), self.vol(J, Iqp)
            self.groups.append((sel, q, r, Iqp, Ipq, Pqp, S, J))

    def vol(self, a, M):
        t = a.reshape(a.shape[:-1] + (M.shape[1],) * self.dim)
        for d in range(self.dim):
            t = _along(t, M, d)
        return t.reshape(a.shape[:-1] + (-1,))

    def face(self, a, M):
        t = a.reshape(a.shape[:-1] + (M.shape[1],) * (self.dim - 1))
        for d in range(self.dim - 1):
            t = _along(t, M, d)
        return t.reshape(a.shape[:-1] + (-1,))

    def boundary(self, uL, N, tag):
        """(ghost state, common state) [K, nv, nfp] at faces of one tag."""
        dim, g1 = self.dim, GAMMA - 1.0
        n = N / N.norm(dim=1, keepdim=True)
        rho, V, pr = uL[:, 0], uL[:, 1:-1] / uL[:, :1], _press(uL)
        if tag == 1:
            mom = uL[:, 1:-1]
            ug, ub = uL.clone(), uL.clone()
            if self.visc:
                ug[:, 1:-1], ub[:, 1:-1] = -mom, 0.0
                ub[:, -1] = uL[:, -1] - 0.5 * (mom ** 2).sum(1) / rho
            else:
                mn = (mom * n).sum(1, keepdim=True)
                ug[:, 1:-1], ub[:, 1:-1] = mom - 2 * mn * n, mom - mn * n
                ub[:, -1] = uL[:, -1] - 0.5 * mn[:, 0] ** 2 / rho
            return ug, ub
        o = self.o
        Vi = torch.tensor(list(o.vel_inf)[:dim], device="cuda", dtype=torch.float64).reshape(1, dim, 1)
        vnL, vnI, cI = (V * n).sum(1), (Vi * n).sum(1), math.sqrt(GAMMA * o.p_inf / o.rho_inf)
        Rp, Rm = vnL + 2 * torch.sqrt(GAMMA * pr / rho) / g1, vnI - 2 * cI / g1
        vn, cb = 0.5 * (Rp + Rm), 0.25 * g1 * (Rp - Rm)
        out = vn > 0
        ent = torch.where(out, pr / rho ** GAMMA, torch.full_like(pr, o.p_inf / o.rho_inf ** GAMMA))
        Vt = torch.where(out[:, None], V - vnL[:, None] * n, Vi - vnI[:, None] * n)
        rb = (cb * cb / (GAMMA * ent)) ** (1.0 / g1)
        Vb = Vt + vn[:, None] * n
        ub = torch.cat([rb[:, None], rb[:, None] * Vb,
                        (rb * cb * cb / GAMMA / g1 + 0.5 * rb * (Vb ** 2).sum(1))[:, None]], 1)
        return ub, ub

    def residual(self, u, src=None, want=False):
        g, dim, p = self.g, self.dim, self.g.p
        E, nv, n = g.E, dim + 2, p + 1
        ref, nf, nfp = g.ref, 2 * dim, n ** (dim - 1)
        ut = u.reshape((E, nv) + (n,) * dim)
        uf = torch.stack([_end(ut, ref.lp if f % 2 else ref.lm, f // 2).reshape(E, nv, nfp) for f in range(nf)], 1)
        pick = lambda a: a.reshape((E * nf,) + a.shape[2:])[g.nb.reshape(-1)].reshape(a.shape)
        uo = pick(uf)
        uc = 0.5 * (uf + uo)
        bc = []
        for tag in (1, 2):
            e, f = torch.nonzero(g.tag == tag, as_tuple=True)
            if len(e):
                ug, ub = self.boundary(uf[e, f], g.N[e, f], tag)
                uo[e, f], uc[e, f] = ug, ub
                bc.append((tag, e, f, ub))
        jmp = uc - uf
        area = g.N.norm(dim=2, keepdim=True)
        nn = (g.N / area).reshape(E * nf, dim, nfp)
        L, Rr = uf.reshape(E * nf, nv, nfp), uo.reshape(E * nf, nv, nfp)
        side = lambda w: ((_fluxes(w, None, 0.0, dim) * nn[:, None]).sum(2), (w[:, 1:-1] * nn).sum(1).abs() / w[:, 0]
                          + torch.sqrt(GAMMA * _press(w) / w[:, 0]))
        (fl, ll), (fr, lr) = side(L), side(Rr)
        Fc = (0.5 * (fl + fr) - 0.5 * torch.maximum(ll, lr)[:, None] * (Rr - L)).reshape(E, nf, nv, nfp) * area
        com = None
        if self.visc:
            own = torch.empty_like(Fc)
            bG = torch.empty((E, nf, nv, dim, nfp), device="cuda", dtype=torch.float64)
            for sel, q, r, Iqp, Ipq, Pqp, S, J in self.groups:
                us, js = (u, jmp) if sel is None else (u[sel], jmp[sel])
                uq, js = (us, js) if q == p else (self.vol(us, Iqp), self.face(js, Pqp))
                K, m = len(us), q + 1
                uq = uq.reshape((K, nv) + (m,) * dim)
                grad = sum((S[:, d] / J[:, None])[:, None] * _along(uq, r.D, d).reshape(K, nv, 1, -1) for d in range(dim))
                gt = grad.reshape((K, nv, dim) + (m,) * dim)
                for f in range(nf):
                    d, lv, h = f // 2, (r.lp if f % 2 else r.lm), (r.hp if f % 2 else r.hm)
                    lc = _end(((S[:, d] / J[:, None]).reshape((K, dim) + (m,) * dim) * _spread(
                        torch.ones((m ** (dim - 1),), device="cuda", dtype=torch.float64), h, d, dim, m)), lv, d)
                    G = _end(gt, lv, d).reshape(K, nv, dim, -1) \
                        + (1.0 if f % 2 else -1.0) * lc.reshape(K, 1, dim, -1) * js[:, f, :, None]
                    G = G if q == p else self.face(G, Ipq)
                    if sel is None:
                        bG[:, f] = G
                    else:
                        bG[sel, f] = G
            for f in range(nf):
                own[:, f] = (_visc(uf[:, f], bG[:, f], self.mu, dim) * g.N[:, f][:, None]).sum(2)
            com = 0.5 * (own - pick(own))
            for tag, e, f, ub in bc:
                w = (_visc(ub, bG[e, f], self.mu, dim) * g.N[e, f][:, None]).sum(2)
                if tag == 1:
                    w[:, -1] = 0.0
                com[e, f] = w
            del bG
            Fc = Fc - com
        R = torch.empty_like(u)
        for sel, q, r, Iqp, Ipq, Pqp, S, J in self.groups:
            us, js, fs = (u, jmp, Fc) if sel is None else (u[sel], jmp[sel], Fc[sel])
            if q < p:
                us, js, fs = self.vol(us, Iqp), self.face(js, Pqp), self.face(fs, Pqp)
            K, m = len(us), q + 1
            ush = us.reshape((K, nv) + (m,) * dim)
            G = None
            if self.visc:
                G = torch.zeros((K, nv, dim, m ** dim), device="cuda", dtype=torch.float64)
                for d in range(dim):
                    qd = _along(ush, r.D, d) + _spread(js[:, 2 * d + 1], r.hp, d, dim, m) - _spread(js[:, 2 * d], r.hm, d, dim, m)
                    G += (S[:, d] / J[:, None])[:, None] * qd.reshape(K, nv, 1, -1)
            Fx = _fluxes(us, G, self.mu, dim)
            div = 0.0
            for d in range(dim):
                Ft = (S[:, d][:, None] * Fx).sum(2).reshape((K, nv) + (m,) * dim)
                cm = fs[:, 2 * d] + _end(Ft, r.lm, d).reshape(K, nv, -1)
                cp = fs[:, 2 * d + 1] - _end(Ft, r.lp, d).reshape(K, nv, -1)
                div = div + _along(Ft, r.D, d) + _spread(cm, r.hm, d, dim, m) + _spread(cp, r.hp, d, dim, m)
            Rq = -div.reshape(K, nv, -1) / J[:, None]
            Rq = Rq if q == p else self.vol(Rq, Ipq)
            if sel is None:
                R = Rq
            else:
                R[sel] = Rq
        if src is not None:
            R[:, -1] += src
        if not want:
            return R
        e, f = torch.nonzero(g.tag == 1, as_tuple=True)
        w = _dev(_gl(n)[1])
        w = (w[:, None] * w).reshape(-1)
        return R, e, ((_press(uf[e, f])[:, None] * g.N[e, f] - com[e, f, 1:-1]) * w).sum(-1)


def _exact_flow(case, seed):
    meshes, opts, dts, u, caps = _flow(case, seed)
    off = np.concatenate([[0], np.cumsum([len(m[0]) for m in meshes])])
    conn = np.concatenate([np.where((m[1][..., :1] >= 0) & (np.arange(3) == 0), m[1] + int(o), m[1])
                           for m, o in zip(meshes, off)])
    g = _Geom(np.concatenate([m[0] for m in meshes]), conn, case["p"])
    s = _Solver(g, opts, caps)
    if case["kind"] == "residual":
        return {"R": s.residual(u)}
    for sel, q, r, Iqp, Ipq, Pqp, S, J in s.groups:   # a state set on an element of lower degree is projected onto it
        if q < case["p"]:
            u[sel] = s.vol(u[sel], Ipq @ Pqp)
    dt = torch.full((g.E, 1, 1), opts.dt, device="cuda", dtype=torch.float64)
    for k in range(len(meshes)):
        if dts is not None:
            dt[off[k]:off[k + 1]] = dts[k]
    mono, t, step = case.get("mesh") == "monopole", MONO_T0, float(opts.dt)
    if mono:
        (A, kk, xs, fr), = C.MONOPOLE_SOURCE
        shape = A * torch.exp(-kk * (_points(meshes[0][0], case["p"]) - torch.tensor(xs, device="cuda")).square().sum(-1))
        hl = (2.0 * g.J[:, None] / g.S.norm(dim=2)).amin(dim=(1, 2))
    if case["kind"] == "poll":
        cand = torch.as_tensor(np.repeat(np.arange(len(meshes)), np.diff(off)), device="cuda")
        fsum, records, surf = 0.0, [[] for _ in meshes], []
        wi = [_lagr(_gl(case["p"] + 1)[0], [x[d] for x in RING]) for d in range(3)]
        wi = _dev(np.einsum("kc,kb,ka->kcba", wi[2], wi[1], wi[0]).reshape(len(RING), -1))
        for k, (nt, nr) in enumerate(_sizes(case)):
            surf.append(_dev(_surface(meshes[k][0], nt, nr, case["nz"])[0] + off[k]))
    for it in range(case["steps"]):
        if mono and case["cfl"] > 0.0:
            V = (u[:, 1:-1] / u[:, :1]).norm(dim=1)
            lam = (V + torch.sqrt(GAMMA * _press(u) / u[:, 0])).amax(dim=1) * (case["p"] + 1) ** 2 / hl
            step = case["cfl"] / float(lam.max())
            dt[:] = step
        if case["kind"] == "poll" and it % case["every"] == 0:
            for k, el in enumerate(surf):
                w = torch.einsum("kn,evn->ekv", wi, u[el]).reshape(-1, 5)
                pr = _press(w[..., None])[:, 0]
                records[k].append(torch.cat([w[:, :1], w[:, 1:4] / w[:, :1], pr[:, None]], 1))
        src = lambda c: shape * math.sin(2 * math.pi * fr * (t + c * step)) if mono else None
        k1 = s.residual(u, src(0.0), want=case["kind"] == "poll")
        if case["kind"] == "poll":
            k1, e, w = k1
            fnow = torch.zeros((len(meshes), 3), device="cuda", dtype=torch.float64).index_add_(0, cand[e], w)
            fsum = fsum + fnow
        k2 = s.residual(u + 0.5 * dt * k1, src(0.5))
        acc = k1 + 2.0 * k2
        k3 = s.residual(u + 0.5 * dt * k2, src(0.5))
        acc = acc + 2.0 * k3
        u = u + dt * (acc + s.residual(u + dt * k3, src(1.0))) / 6.0
        t += step
    got = {"u": u}
    if case["kind"] == "poll":
        qa = 0.5 * opts.rho_inf * sum(v * v for v in opts.vel_inf) * opts.ref_area
        dirs = torch.tensor([list(opts.lift_dir), list(opts.drag_dir)], device="cuda", dtype=torch.float64)
        now, mean = fnow @ dirs.T / qa, fsum @ dirs.T / (qa * case["steps"])
        got["forces"] = torch.cat([now, mean, torch.full_like(now[:, :1], case["steps"])], 1).cpu().numpy()
        got["records"] = [torch.stack(r).cpu().numpy() for r in records]
    return got


def _exact_fwh(case, seed):
    r = _fwh_inputs(case, seed)
    M, c0, dt, nt = torch.tensor(r["M"], device="cuda", dtype=torch.float64), r["c0"], r["dt"], case["nt"]
    U = c0 * M
    h, n = r["hist"], r["n"]
    Un = n @ U
    vn = (h[..., 1:4] * n).sum(-1)                                # total normal velocity = u_n + U_n
    Q = h[..., 0] * vn - Un
    Lm = (h[..., 4:5] - r["p0"]) * n + (h[..., 0] * vn)[..., None] * (h[..., 1:4] - U)
    X = torch.cat([Q[..., None], Lm], -1).permute(1, 2, 0).contiguous()     # [npts, 4, nt]
    dX = torch.empty_like(X)
    dX[..., 2:-2] = X[..., :-4] - 8 * X[..., 1:-3] + 8 * X[..., 3:-1] - X[..., 4:]
    for t, j0, c in ((0, 0, (-25, 48, -36, 16, -3)), (1, 0, (-3, -10, 18, -6, 1)),
                     (nt - 2, nt - 5, (-1, 6, -18, 10, 3)), (nt - 1, nt - 5, (3, -16, 36, -48, 25))):
        dX[..., t] = sum(c[m] * X[..., j0 + m] for m in range(5))
    X = torch.cat([X, dX / (12 * dt)], 1)                         # Q, L, dQ, dL
    b2 = 1.0 / (1.0 - float(M @ M))
    K = case["copies"] // 2
    out = torch.zeros((case["obs"], nt), device="cuda", dtype=torch.float64)
    T, t0 = [], []
    for o, at in enumerate(_dev(r["obs"])):
        geo = []
        for k in range(-K, K + 1):
            y = r["y"].clone()
            y[:, 2] += 0.2 * k
            d = at - y
            Mr = d @ M
            Rs = torch.sqrt((d * d).sum(1) + b2 * Mr * Mr) / math.sqrt(b2)
            R = b2 * (Rs - Mr)
            dRs = (d + b2 * Mr[:, None] * M) / (b2 * Rs[:, None])
            dR = b2 * (dRs - M)
            cf = torch.cat([(-c0 * (dRs @ M) / Rs ** 2)[:, None], dRs / Rs[:, None] ** 2,
                            ((1.0 - dR @ M) / Rs)[:, None], dR / (c0 * Rs[:, None])], 1) * r["dS"][:, None]
            geo.append((cf, R / c0))
        lo, hi = max(float(g[1].max()) for g in geo), min(float(g[1].min()) for g in geo)
        Tn = int(math.floor(((nt - 1) * dt + hi - lo) / dt + 1e-9)) + 1
        i = torch.arange(Tn, device="cuda", dtype=torch.float64)
        for cf, delay in geo:
            I = (cf[:, :, None] * X).sum(1)
            pos = i + ((lo - delay) / dt)[:, None]
            j = (pos.floor().long() - 1).clamp(0, nt - 4)
            x = pos - j
            for m, w in enumerate((-(x - 1) * (x - 2) * (x - 3) / 6, x * (x - 2) * (x - 3) / 2,
                                   -x * (x - 1) * (x - 3) / 2, x * (x - 1) * (x - 2) / 6)):
                out[o, :Tn] += (w * I.gather(1, j + m)).sum(0)
        T.append(Tn)
        t0.append(lo)
    out /= 4 * math.pi
    m = min(T)
    L = 2 * (m // (case["nseg"] + 1))
    win = 0.5 - 0.5 * torch.cos(2 * math.pi * torch.arange(L, device="cuda", dtype=torch.float64) / L)
    seg = torch.stack([out[:, k * (L // 2):k * (L // 2) + L] for k in range(case["nseg"])], 1)
    P = torch.fft.rfft((seg - seg.mean(-1, keepdim=True)) * win).abs().square().mean(1) * dt / win.square().sum()
    P[:, 1:L // 2] *= 2.0
    return {"p": out, "nt": None, "t0": np.array(t0), "psd": P, "freq": np.arange(L // 2 + 1) / (L * dt)}


def exact(case, seed):
    return _exact_fwh(case, seed) if case["kind"] == "fwh" else _exact_flow(case, seed)
