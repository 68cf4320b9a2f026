"""Performance cases of the phase-field lattice Boltzmann library: what a user's
program has it do, through the public Python binding.

A pass advances a simulation by a number of time steps and reads the result
back, as a run does between two outputs: the five fields into pinned host
arrays, or the checkpoint.  A pass continues from the state that the previous
one left.  The kinds:

  drop      static droplet, periodic (the Laplace-law workload)
  layer     layered Poiseuille flow between walls, step viscosity, body force
  spinodal  phase separation of a noisy mixture, periodic
  impact    droplet impact on a film, walls or an open top, the spreading
            radius read several times on the way
  batch     many uneven drops and impacts advanced together
"""
import math

import numpy as np
import torch

from paper_1710_09541_gb300 import cases as inputs
from paper_1710_09541_gb300 import lbm

STORAGE = {"fp32": lbm.LBM_STORE_FP32, "fp16": lbm.LBM_STORE_FP16_SHIFTED,
           "bf16": lbm.LBM_STORE_BF16_SHIFTED, "bf16_sr": lbm.LBM_STORE_BF16_SHIFTED_SR}
FIELDS = ("phi", "rho", "ux", "uy", "p")


def listed():
    return [
        # the smallest grid a user runs: the Laplace-law droplet, bound by latency and launches
        dict(name="drop64", kind="drop", nx=64, ny=64, storage="fp32", steps=100, normal=0, out="fields"),
        # layered Poiseuille flow on its narrow walled grid (run for 1e5 steps to reach steady state)
        dict(name="layer8x256", kind="layer", nx=8, ny=256, storage="fp32", steps=200, normal=0, out="fields"),
        # the droplet of the paper's Sec. III A with its own normal (Eq. 29), ended by a checkpoint
        dict(name="drop200_eq29_ckpt", kind="drop", nx=200, ny=200, storage="fp32", steps=100, normal=1, out="state"),
        # an ordinary grid of odd sizes with an open top, finiteness checks on, odd step count
        dict(name="impact701x333_open", kind="impact", nx=701, ny=333, storage="fp32", steps=77, normal=0, bc=2,
             check_every=20, calls=1, out="fields"),
        # spinodal decomposition, the phase-separation workload, in both storage formats it is run in
        dict(name="spinodal1024", kind="spinodal", nx=1024, ny=1024, storage="fp32", steps=100, normal=0, out="fields"),
        dict(name="spinodal1024_fp16", kind="spinodal", nx=1024, ny=1024, storage="fp16", steps=100, normal=0,
             out="fields"),
        # droplet impact: walls, the spreading radius sampled on the way
        dict(name="impact2400x600", kind="impact", nx=2400, ny=600, storage="fp32", steps=100, normal=0, bc=1,
             check_every=0, calls=4, out="fields"),
        dict(name="impact2400x600_bf16", kind="impact", nx=2400, ny=600, storage="bf16", steps=100, normal=0, bc=1,
             check_every=0, calls=4, out="fields"),
        # an odd-sized periodic grid in the stochastically rounded format
        dict(name="spinodal1501x1103_sr", kind="spinodal", nx=1501, ny=1103, storage="bf16_sr", steps=61, normal=0,
             out="fields"),
        # the throughput workload, 2048 x 2048 periodic, in FP32 and FP16 storage
        dict(name="spinodal2048", kind="spinodal", nx=2048, ny=2048, storage="fp32", steps=100, normal=0, out="fields"),
        dict(name="spinodal2048_fp16", kind="spinodal", nx=2048, ny=2048, storage="fp16", steps=100, normal=0,
             out="fields"),
        # the sweep: 64 uneven cases in one batch, FP16 storage
        dict(name="batch64_fp16", kind="batch", cases=64, pick=7, storage="fp16", steps=160, out="fields"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["drop", "drop", "layer", "spinodal", "spinodal", "impact", "impact", "batch"])
    storage = rng.choice(["fp32", "fp32", "fp16", "fp16", "bf16", "bf16_sr"])
    if kind == "batch":
        storage = rng.choice(["fp32", "fp16", "fp16", "bf16"])
        return dict(kind=kind, cases=_log(rng, 2, 32 if storage == "fp32" else 54), pick=rng.randrange(1, 1 << 20),
                    storage=storage, steps=rng.randint(140, 160), out="fields")
    c = dict(kind=kind, storage=storage, steps=_log(rng, 20, 200), normal=rng.choice([0, 0, 1]), out="fields")
    if kind == "layer":
        c.update(nx=_log(rng, 4, 64), ny=_log(rng, 64, 512), normal=0, storage="fp32")
    elif kind == "drop":
        c.update(nx=_log(rng, 48, 1024), ny=_log(rng, 48, 1024), out=rng.choice(["fields", "fields", "state"]))
    elif kind == "spinodal":
        c.update(nx=_log(rng, 96, 2048), ny=_log(rng, 96, 2048))
    else:
        c.update(nx=_log(rng, 240, 2400), ny=_log(rng, 120, 1200), bc=rng.choice([1, 2]),
                 check_every=rng.choice([0, 0, 25]), calls=rng.randint(1, 5),
                 storage=rng.choice(["fp32", "fp16", "bf16"]))
    return c


def _problem(case, seed):
    """(params, phi0, ux0, uy0) of a single case: the workloads' own recipes,
    with positions, radii or noise from the seed."""
    nx, ny, kind = case["nx"], case["ny"], case["kind"]
    u = inputs.uniform01(1000 * (seed % (1 << 40)) + 17, 4)
    if kind == "drop":
        P = inputs.params_static_drop()
        R = 0.25 * min(nx, ny) * (0.9 + 0.1 * u[0])
        return P, inputs.drop(nx, ny, R, P["W"], x0=nx / 2 + 4 * u[1], y0=ny / 2 + 4 * u[2]), None, None
    if kind == "layer":
        P = inputs.params_poiseuille(ny)
        return P, inputs.layer(nx, ny, P["W"], y_if=ny / 2 + 4 * (u[0] - 0.5)), None, None
    if kind == "spinodal":
        return inputs.params_spinodal(), inputs.spinodal(nx, ny, seed=seed % (1 << 40)), None, None
    D = min(200.0, 0.3 * min(nx, ny)) * (0.95 + 0.05 * u[0])
    P = dict(inputs.params_impact(D=D, Re=100.0), bc_y=case["bc"])
    return (P, *inputs.impact(nx, ny, D, 0.1 * D, 0.04, P["W"]))


def _batch_problems(case, seed):
    specs = inputs.batch_cases(case["cases"], seed=case["pick"])
    u = inputs.uniform01(1000 * (seed % (1 << 40)) + 29, len(specs))
    for s, v in zip(specs, u):  # each case's order parameter shifted along x by its own distance
        k = int(v * s["nx"])
        for a in ("phi0", "ux0", "uy0"):
            s[a] = np.roll(s[a], k, axis=1)
    return specs


def _pinned(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True)


def prepare(case, seed):
    storage = STORAGE[case["storage"]]
    if case["kind"] == "batch":
        lats, total = [], 0
        for s in _batch_problems(case, seed):
            lat = lbm.Lattice(s["nx"], s["ny"], storage=storage, **s["params"])
            lats.append(lat.init(s["phi0"], s["ux0"], s["uy0"]))
            total += s["nx"] * s["ny"]
        host = _pinned((5 * total,))
        views, at = [], 0
        flat = host.numpy()
        for lat in lats:  # each case's five fields, one after the other
            n = lat.nx * lat.ny
            views.append({k: flat[at + j * n:at + (j + 1) * n].reshape(lat.ny, lat.nx) for j, k in enumerate(FIELDS)})
            at += 5 * n
        return dict(case=case, batch=lbm.Batch(lats), lats=lats, host=host, views=views)
    P, phi0, ux0, uy0 = _problem(case, seed)
    lat = lbm.Lattice(case["nx"], case["ny"], storage=storage, normal_scheme=case["normal"],
                      check_every=case.get("check_every", 0), **P)
    lat.init(phi0, ux0, uy0)
    host = _pinned((5, case["ny"], case["nx"]))
    return dict(case=case, lat=lat, host=host, views=dict(zip(FIELDS, host.numpy())))


def _sample_steps(case):
    """steps of each call of an impact run (the radius is read after each)"""
    n, k = case["steps"], case["calls"]
    return [(j + 1) * n // k - j * n // k for j in range(k)]


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        for lat, out in zip(state["lats"], state["views"]):
            lat.fields(out=out)
        return state["host"]
    lat, radii = state["lat"], []
    if case["kind"] == "impact":
        for n in _sample_steps(case):
            lat.step(n)
            radii.append(lat.spreading_radius(lat.ny // 10)[0])
    else:
        lat.step(case["steps"])
    if case["out"] == "state":
        return dict(zip(("f", "g", "phiu"), lat.get_state()))
    lat.fields(out=state["views"])
    return {"fields": dict(zip(FIELDS, state["host"])), "radii": radii} if radii else dict(zip(FIELDS, state["host"]))


# Floating-point operations that one node needs in one step: the moments of f
# and g (8 + 27), the stencils (34), the recovery of rho, mu, F, u, p (34), the
# relaxation and source terms (40), nine Allen-Cahn (5 each) and nine
# Navier-Stokes (11 each) updates.
FLOPS = 8 + 27 + 34 + 34 + 40 + 9 * 5 + 9 * 11


def work(case):
    """One pass reads the state once, writes it once, and writes the output:
    18 populations and (phi u) of a node, as the storage format keeps them
    (80 or 46 bytes), and five doubles or a checkpoint of 20 floats."""
    if case["kind"] == "batch":
        n = sum(s["nx"] * s["ny"] for s in _sizes(case))
    else:
        n = case["nx"] * case["ny"]
    state = 80 if case["storage"] == "fp32" else 46
    return {"bytes": n * (2 * state + (80 if case["out"] == "state" else 40)), "flops": n * case["steps"] * FLOPS}


def _sizes(case):
    u = inputs.uniform01(case["pick"], 6 * case["cases"]).reshape(case["cases"], 6)
    return [dict(nx=256 + 64 * int(r[0] * 13), ny=256 + 64 * int(r[1] * 5)) for r in u]


# ---- the model in 64 bits ------------------------------------------------------
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


class _Model:
    """Sec. II of arXiv:1710.09541 on FP64 tensors [ny, nx]; f, g are the
    pre-collision populations."""

    def __init__(self, P, normal, phi0, ux0, uy0):
        t = lambda a: (torch.zeros(phi0.shape, dtype=torch.float64, device="cuda") if a is None  # noqa: E731
                       else torch.as_tensor(np.ascontiguousarray(a), device="cuda"))
        self.P, self.normal, self.bc = P, normal, P["bc_y"]
        phi, ux, uy = t(phi0), t(ux0), t(uy0)
        rho = phi * (P["rho_l"] - P["rho_g"]) + P["rho_g"]
        usq = ux * ux + uy * uy
        self.f, self.g = [], []
        for i in range(9):
            cu = CX[i] * ux + CY[i] * uy
            self.f.append(WT[i] * phi * (1 + 3 * cu))
            self.g.append(rho * WT[i] * (3 * cu + 4.5 * cu * cu - 1.5 * usq))
        self.phiux, self.phiuy = phi * ux, phi * uy
        self._top()

    def _top(self):
        if self.bc == 2:  # open top: the entering populations repeat the row below
            for i in (4, 7, 8):
                for s in (self.f, self.g):
                    s[i] = s[i].clone()
                    s[i][-1] = s[i][-2]

    def _shift(self, a, dx, dy):
        """a(x + dx, y + dy), periodic in x, periodic or edge-repeating in y"""
        if dy:
            if self.bc == 0:
                a = torch.roll(a, -dy, 0)
            else:
                a = torch.cat([a[1:], a[-1:]]) if dy > 0 else torch.cat([a[:1], a[:-1]])
        return torch.roll(a, -dx, 1) if dx else a

    def macro(self):
        P = self.P
        phi = sum(self.f[1:], self.f[0])
        gx, gy, lap = torch.zeros_like(phi), torch.zeros_like(phi), torch.zeros_like(phi)
        for i in range(1, 9):
            d = self._shift(phi, CX[i], CY[i])
            gx += 3 * WT[i] * CX[i] * d
            gy += 3 * WT[i] * CY[i] * d
            lap += 6 * WT[i] * (d - phi)
        drho = P["rho_l"] - P["rho_g"]
        rho = phi * drho + P["rho_g"]
        k, beta = 1.5 * P["sigma"] * P["W"], 12 * P["sigma"] / P["W"]
        mu = 4 * beta * phi * (phi - 1) * (phi - 0.5) - k * lap
        Fx, Fy = mu * gx + P["Gx"], mu * gy + P["Gy"]
        mx = sum(CX[i] * self.g[i] for i in range(1, 9) if CX[i])
        my = sum(CY[i] * self.g[i] for i in range(1, 9) if CY[i])
        ux, uy = (mx + 0.5 * Fx) / rho, (my + 0.5 * Fy) / rho
        usq = ux * ux + uy * uy
        p = 0.6 * (sum(self.g[2:], self.g[1]) + 0.5 * drho * (ux * gx + uy * gy) - 2 / 3 * rho * usq)
        return phi, rho, ux, uy, p, usq, gx, gy, Fx, Fy

    def step(self):
        P = self.P
        phi, rho, ux, uy, p, usq, gx, gy, Fx, Fy = self.macro()
        drho = P["rho_l"] - P["rho_g"]
        if P["visc_mode"] == 2:
            nu = torch.where(phi >= 0.5, P["rho_l"] * P["nu_l"], P["rho_g"] * P["nu_g"]) / rho
        else:
            nu = phi * (P["nu_l"] - P["nu_g"]) + P["nu_g"]
        tau = 3 * nu + 0.5
        pux, puy = phi * ux, phi * uy
        Dx, Dy = pux - self.phiux, puy - self.phiuy
        self.phiux, self.phiuy = pux, puy
        if self.normal == 0:
            nx, ny = gx, gy
        else:
            nx, ny = 0.5 * Dx, 0.5 * Dy
            for i in range(1, 9):
                ne = self.f[i] - WT[i] * phi * (1 + 3 * (CX[i] * ux + CY[i] * uy))
                nx, ny = nx + CX[i] * ne, ny + CY[i] * ne
            nx, ny = -nx, -ny
        n2 = nx * nx + ny * ny
        inv = torch.where(n2 > 1e-12, 1 / torch.sqrt(torch.clamp(n2, min=1e-300)), torch.zeros_like(n2))
        lam = 4 / P["W"] * phi * (1 - phi)
        Sx, Sy = Dx + lam * nx * inv / 3, Dy + lam * ny * inv / 3
        tf = P["tau_h"]
        pf, pg = [], []
        for i in range(9):
            cu = CX[i] * ux + CY[i] * uy
            feq = WT[i] * phi * (1 + 3 * cu)
            F = (1 - 0.5 / tf) * WT[i] * 3 * (CX[i] * Sx + CY[i] * Sy)
            pf.append(self.f[i] - (self.f[i] - feq) / tf + F)
            geq = 3 * p * (WT[i] - (i == 0)) + rho * WT[i] * (3 * cu + 4.5 * cu * cu - 1.5 * usq)
            G = (1 - 0.5 / tau) * WT[i] * 3 * (CX[i] * Fx + CY[i] * Fy + drho * cu * (CX[i] * gx + CY[i] * gy))
            pg.append(self.g[i] - (self.g[i] - geq) / tau + G)
        for i in range(9):
            for s, q in ((self.f, pf), (self.g, pg)):
                a = torch.roll(q[i], (CY[i], CX[i]), (0, 1))
                if self.bc and CY[i] == 1:
                    a[0] = q[OPP[i]][0]
                elif self.bc == 1 and CY[i] == -1:
                    a[-1] = q[OPP[i]][-1]
                s[i] = a
        self._top()


def _radius(phi, xc):
    """half the extent of the run of phi >= 1/2 through column xc of a row"""
    wet = (phi >= 0.5).cpu().numpy()
    if not wet[xc]:
        return 0.0
    dry = np.flatnonzero(~wet)
    left, right = dry[dry < xc], dry[dry > xc]
    return 0.5 * ((right[0] if right.size else wet.size) - (left[-1] if left.size else -1) - 1)


def exact(case, seed):
    if case["kind"] == "batch":
        # a 16-bit case's velocity and pressure have no 64-bit counterpart close
        # enough to be told from another's, and they share one array with the
        # order parameter
        if case["storage"] != "fp32":
            return None
        out = []
        for s in _batch_problems(case, seed):
            m = _Model(s["params"], 0, s["phi0"], s["ux0"], s["uy0"])
            for _ in range(case["steps"]):
                m.step()
            out += [a.reshape(-1) for a in m.macro()[:5]]
        return torch.cat(out)
    P, phi0, ux0, uy0 = _problem(case, seed)
    m = _Model(P, case["normal"], phi0, ux0, uy0)
    radii = []
    for n in _sample_steps(case) if case["kind"] == "impact" else [case["steps"]]:
        for _ in range(n):
            m.step()
        radii.append(_radius(sum(m.f[1:], m.f[0])[case["ny"] // 10], case["nx"] // 2))
    fp32 = case["storage"] == "fp32"
    if case["out"] == "state":
        # the codes of the 16-bit formats hold g with 8 or 11 bits: only f is near its 64-bit value
        return {"f": torch.stack(m.f), "g": torch.stack(m.g) if fp32 else None,
                "phiu": torch.stack([m.phiux, m.phiuy]) if fp32 else None}
    # with 16-bit storage u and p carry the rounding of g; phi and rho are near their 64-bit values
    fields = {k: a if fp32 or k in ("phi", "rho") else None for k, a in zip(FIELDS, m.macro()[:5])}
    return {"fields": fields, "radii": radii} if case["kind"] == "impact" else fields
