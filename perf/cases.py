"""Performance cases: what a user of the black-oil library has it do.

Every case goes through the public Python entry points (``Sim``, ``Ensemble``)
and returns whole results: states, rates, Newton corrections, products.  The
models are the repository's own shapes (the SPE1-shaped 10x10x3 model, the
ensemble's 20..64 x 20..64 x 5..16 members, the 100x100x50 GRF model, the
60x220x85 layered model) with fields drawn from the seed, and a state part way
through a flood: water around the injectors, free gas in places, pressure near
the oil column's.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1910_06059_gb300 import Ensemble, Sim
from synth.models import DAY, FT, MD, MSCF, PSI, STB, fluid_params

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one field-scale sub-step of the SPE1-shaped model (coarse cells, a gas
        # injector): the smallest model, where launches and round trips count
        {"name": "spe1_step", "kind": "step", "model": "spe1", "nx": 10, "ny": 10, "nz": 3,
         "days": 1.0, "precond": "ilu0", "wells": "reduced", "ysub": 0, "zsub": 0},
        # a small history-matching member on its own, default solver
        {"name": "member_ilu0_step", "kind": "step", "model": "member", "nx": 33, "ny": 27,
         "nz": 9, "days": 0.01, "precond": "ilu0", "wells": "reduced", "ysub": 0, "zsub": 0},
        # a large member with the preconditioner the ensembles use
        {"name": "member_cpr_step", "kind": "step", "model": "member", "nx": 61, "ny": 58,
         "nz": 15, "days": 0.01, "precond": "cpr", "wells": "reduced", "ysub": 0, "zsub": 0},
        # the full standard well (four unknowns, cross-flow, storage) on a ragged grid
        {"name": "std_wells_step", "kind": "step", "model": "grf", "nx": 47, "ny": 53, "nz": 21,
         "days": 0.01, "precond": "cpr", "wells": "standard", "ysub": 0, "zsub": 0},
        # a sub-step of the 500,000-cell GRF model, default solver
        {"name": "grf_ilu0_step", "kind": "step", "model": "grf", "nx": 100, "ny": 100, "nz": 50,
         "days": 0.003, "precond": "ilu0", "wells": "reduced", "ysub": 0, "zsub": 0},
        # half of the layered model with an odd number of layers, CPR
        {"name": "half_cpr_step", "kind": "step", "model": "layered", "nx": 60, "ny": 110,
         "nz": 43, "days": 0.003, "precond": "cpr", "wells": "reduced", "ysub": 0, "zsub": 0},
        # the benchmark model, default solver: a Newton loop driven by the caller
        # (linearise, test, solve, update)
        {"name": "layered_ilu0_newton", "kind": "newton", "model": "layered", "nx": 60, "ny": 220,
         "nz": 85, "days": 0.05, "precond": "ilu0", "wells": "reduced", "ysub": 0, "zsub": 0,
         "iterations": 3},
        # the same with the fastest configuration: CPR, boxes in its second stage
        {"name": "layered_cpr_newton", "kind": "newton", "model": "layered", "nx": 60, "ny": 220,
         "nz": 85, "days": 0.02, "precond": "cpr", "wells": "reduced", "ysub": 56, "zsub": 44,
         "iterations": 4},
        # an external Krylov method's operator and preconditioner products on host vectors
        {"name": "products", "kind": "products", "model": "grf", "nx": 51, "ny": 49, "nz": 25,
         "days": 0.5, "precond": "ilu0", "wells": "reduced", "ysub": 0, "zsub": 0},
        # uneven members of a history-matching ensemble stepped together
        {"name": "ensemble_cpr", "kind": "ensemble", "members": 24, "lo": 20, "hi": 64,
         "days": 0.01, "precond": "cpr"},
    ]


def draw(rng):
    """One more case of the same ranges."""
    def size(lo, hi):   # log-uniform integer
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def days(lo, hi):
        return round(math.exp(rng.uniform(math.log(lo), math.log(hi))), 4)

    pick = rng.choice(["small", "small", "member", "member", "field", "field", "newton",
                       "products", "ensemble"])
    c = {"kind": "step", "precond": rng.choice(["ilu0", "cpr"]), "wells": "reduced", "ysub": 0,
         "zsub": 0}
    if pick == "small":
        c.update(model="spe1", nx=size(6, 24), ny=size(6, 24), nz=rng.randint(2, 6),
                 days=days(0.3, 2.0))
    elif pick == "member":
        c.update(model="member", nx=size(20, 64), ny=size(20, 64), nz=rng.randint(5, 16),
                 days=days(0.003, 0.01), wells=rng.choice(["reduced", "reduced", "standard"]))
    elif pick == "field":
        c.update(model=rng.choice(["grf", "layered"]), nx=size(30, 100), ny=size(40, 130),
                 nz=size(10, 50), days=days(0.001, 0.003))
        if c["precond"] == "cpr" and rng.random() < 0.5:
            c.update(ysub=8 * rng.randint(3, 7), zsub=4 * rng.randint(3, 8))
    elif pick == "newton":
        c.update(kind="newton", model="layered", nx=size(20, 60), ny=size(30, 110),
                 nz=size(8, 43), days=days(0.005, 0.05), iterations=rng.randint(1, 4))
    elif pick == "products":
        c.update(kind="products", model="grf", nx=size(16, 64), ny=size(16, 64), nz=size(5, 32),
                 days=days(0.1, 1.0))
    else:
        c = {"kind": "ensemble", "members": rng.randint(8, 20), "lo": 20,
             "hi": rng.randint(32, 64), "days": days(0.003, 0.01), "precond": "cpr"}
    return c


# ---------------------------------------------------------------------------
# Models and states
# ---------------------------------------------------------------------------
def _well(i, j, ks, kind, control, target, limit, phase="gas"):
    return {"i": int(i), "j": int(j), "ks": [int(k) for k in ks], "kind": kind, "phase": phase,
            "control": control, "target": float(target), "bhp_limit": float(limit), "rw": 0.1,
            "skin": 0.0}


def _grf(g, shape, corr):
    """Unit-variance Gaussian field on the device over the last len(corr)
    axes (spectral method, twice padded), independent along the others."""
    d = len(corr)
    pad = list(shape[:-d]) + [2 * v for v in shape[-d:]]
    white = torch.randn(pad, generator=g, device=DEV, dtype=F64)
    k2 = 0.0
    for a, c in enumerate(corr):
        f = (c * torch.fft.fftfreq(pad[len(pad) - d + a], device=DEV, dtype=F64)) ** 2
        k2 = k2 + f.reshape([-1 if b == a else 1 for b in range(d)])
    axes = tuple(range(-d, 0))
    f = torch.fft.ifftn(torch.fft.fftn(white, dim=axes) * torch.exp(-0.5 * math.pi ** 2 * k2),
                        dim=axes).real
    f = f[tuple(slice(0, v) for v in shape)]
    f = f - f.mean(dim=axes, keepdim=True)
    return f / f.std(dim=axes, keepdim=True).clamp_min(1e-12)


def _model(case, g):
    """(model dict, ln k field on the device) of the case."""
    nx, ny, nz, kind = case["nx"], case["ny"], case["nz"], case["model"]
    mean = math.log(200 * MD)
    ks = list(range(nz))
    dx, dy, dz = 20 * FT, 10 * FT, 2 * FT
    if kind == "spe1":
        lnk = mean + torch.randn((nz, ny, nx), generator=g, device=DEV, dtype=F64)
        poro = torch.full_like(lnk, 0.3)
        dx, dy, dz = 1000 * FT, 1000 * FT, 50 * FT
        wells = [_well(0, 0, [0], "inj", "rate", 100e3 * MSCF / DAY, 9014 * PSI),
                 _well(nx - 1, ny - 1, [nz - 1], "prod", "bhp", 1000 * PSI, 1000 * PSI)]
    else:
        if kind == "member":
            sigma = 1.5
            lnk = mean + sigma * _grf(g, (nz, ny, nx), (8.0, 8.0, 8.0))
        elif kind == "grf":
            sigma = 1.5
            lnk = mean + sigma * _grf(g, (nz, ny, nx), (10.0, 10.0, 10.0))
        else:                                 # layered: channels in the odd layers
            sigma = 2.0
            lnk = mean + sigma * _grf(g, (nz, ny, nx), (8.0, 8.0))
            u = torch.rand((3, nz, 1, 1), generator=g, device=DEV, dtype=F64)
            th, lam = (20 + 40 * u[0]) * math.pi / 180, 20 + 40 * u[1]
            y, x = torch.meshgrid(torch.arange(ny, device=DEV, dtype=F64),
                                  torch.arange(nx, device=DEV, dtype=F64), indexing="ij")
            band = torch.sin(2 * math.pi * (x * torch.cos(th) + y * torch.sin(th)) / lam
                             + 2 * math.pi * u[2]).abs() > 0.8
            band[0::2] = False
            lnk = lnk + 3.0 * band
        poro = (0.2 + 0.05 * (lnk - mean) / sigma).clamp(0.05, 0.35)
        if kind == "member":
            rate = 0.002 * float(poro.sum()) * dx * dy * dz / DAY
            wells = [_well(0, 0, ks, "inj", "rate", rate, 10000 * PSI, "water"),
                     _well(nx - 1, ny - 1, ks, "prod", "bhp", 3000 * PSI, 3000 * PSI)]
        else:
            # the five-spot's 5000 stb/day of the benchmark model, per pore volume
            rate = 5000 * STB / DAY * min(1.0, nx * ny * nz / 500_000)
            wells = [_well(nx // 2, ny // 2, ks, "inj", "rate", rate, 10000 * PSI, "water")]
            wells += [_well(i, j, ks, "prod", "bhp", 3000 * PSI, 3000 * PSI)
                      for j in (0, ny - 1) for i in (0, nx - 1)]
    m = {"name": kind, "nx": nx, "ny": ny, "nz": nz, "dx": np.full(nx, dx),
         "dy": np.full(ny, dy), "dz": np.full(nz, dz), "top_depth": 2500.0,
         "perm": torch.exp(lnk).reshape(-1).cpu().numpy(),
         "poro": poro.reshape(-1).cpu().numpy(), "fluid": fluid_params(), "wells": wells,
         "init": {"p_top": 4800.0 * PSI, "sw": 0.15, "rgo": 180.0}}
    return m


def _state(m, g):
    """A state part way through a flood, on the device: (p, sw, x, flag, bhp).
    Pressure drawn down around the producers, below the bubble point next to
    them, where the oil has lost its gas; water around the injectors."""
    nx, ny, nz = m["nx"], m["ny"], m["nz"]
    a, b = (_grf(g, (nz, ny, nx), (2.0, 6.0, 6.0)) for _ in range(2))
    f = m["fluid"]
    dz = torch.as_tensor(m["dz"], device=DEV, dtype=F64)
    z = (torch.cumsum(dz, 0) - 0.5 * dz)[:, None, None]
    y, x = torch.meshgrid(torch.arange(ny, device=DEV, dtype=F64),
                          torch.arange(nx, device=DEV, dtype=F64), indexing="ij")
    p = 4800 * PSI + 700.0 * f["g"] * (z - z[0]) + 2 * PSI * a
    sw = 0.15 + 0.01 * torch.sigmoid(b)
    for w in m["wells"]:
        near = torch.exp(-torch.hypot(x - w["i"], y - w["j"]) / (1.0 + 0.1 * min(nx, ny)))
        p = p + ((200 * PSI) if w["kind"] == "inj" else (-1000 * PSI)) * near
        if w["kind"] == "inj" and w["phase"] == "water":
            sw = sw + 0.35 * near * torch.sigmoid(b + 1.0)
    r = 170.0 + 2.0 * torch.tanh(b)
    ps = f["p_b"] / f["R_sb"] * r                   # saturation pressure of the oil
    sat = p < ps
    x = torch.where(sat, 0.5 * (1 - p / ps), r)
    bhp = [w["target"] if w["control"] == "bhp" else 5500 * PSI for w in m["wells"]]
    return (p.reshape(-1).contiguous(), sw.reshape(-1).contiguous(), x.reshape(-1).contiguous(),
            (~sat).to(torch.uint8).reshape(-1).contiguous(),
            torch.tensor(bhp, device=DEV, dtype=F64))


def _configure(sim, case):
    if case.get("wells") == "standard":
        sim.set_well_model("standard", storage=True)
    if case["precond"] != "ilu0":
        sim.preconditioner = case["precond"]
    if case.get("ysub"):
        sim.subdomains = case["ysub"]
    if case.get("zsub"):
        sim.subdomains_z = case["zsub"]


def _members(case):
    """The uneven members of an ensemble case, as single-model cases; member
    q's size depends on q alone, its fields on the seed."""
    out = []
    for q in range(case["members"]):
        r = random.Random(q)
        out.append({"model": "member", "nx": r.randint(case["lo"], case["hi"]),
                    "ny": r.randint(case["lo"], case["hi"]), "nz": r.randint(5, 16)})
    return out


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    if case["kind"] == "ensemble":
        models = [_model(c, g) for c in _members(case)]
        states = [_state(m, g) for m in models]
        ens = Ensemble(models, streams=64)
        for s in ens.members:
            _configure(s, case)
        return {"case": case, "ens": ens, "states": states}
    m = _model(case, g)
    state = _state(m, g)
    sim = Sim(m)
    _configure(sim, case)
    out = {"case": case, "sim": sim, "state": state}
    if case["kind"] == "products":
        sim.set_state_dev(*state)
        sim.begin_step()
        sim.assemble(case["days"] * DAY)
        sim.factor()
        scale = torch.tensor([1e5, 0.05, 0.05], device=DEV, dtype=F64)
        v = torch.randn((sim.n, 3), generator=g, device=DEV, dtype=F64)
        out["v"] = (v * scale).reshape(-1).cpu().numpy()
    return out


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _read_state(sim):
    p, sw, x = (torch.empty(sim.n, device=DEV, dtype=F64) for _ in range(3))
    flag = torch.empty(sim.n, device=DEV, dtype=torch.uint8)
    bhp = torch.empty(sim.nw, device=DEV, dtype=F64)
    sim.get_state_dev(p, sw, x, flag, bhp)
    return {"p": p, "sw": sw, "x": x, "flag": flag, "bhp": bhp}


def run(state):
    case = state["case"]
    dt = case["days"] * DAY
    if case["kind"] == "ensemble":
        ens = state["ens"]
        for s, v in zip(ens.members, state["states"]):
            s.set_state_dev(*v)
            s.dt_next = dt
        ens.step(dt, raise_on_fail=False)
        # the states of all members side by side, member after member
        outs = [_read_state(s) for s in ens.members]
        return {k: torch.cat([o[k] for o in outs]) for k in outs[0]}
    sim = state["sim"]
    if case["kind"] == "products":
        return {"op": sim.apply_op(state["v"]), "prec": sim.precond_apply(state["v"])}
    sim.set_state_dev(*state["state"])
    if case["kind"] == "newton":
        sim.begin_step()
        out = {}
        for q in range(case["iterations"]):
            sim.assemble(dt)
            out["norms%d" % q] = sim.norms(dt)
            _, _, out["sol%d" % q] = sim.solve()
            sim.newton_update()
        return {**out, **_read_state(sim)}
    sim.dt_next = dt
    sim.step(dt)
    return {**_read_state(sim), "rates": sim.well_rates()[0]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
# Typical Newton iterations of a pass (of the coarse SPE1-shaped cells, of the
# others) and BiCGStab iterations of a solve (of a short sub-step, of a long one).
_NEWTON = {"spe1": 4, "step": 12, "ensemble": 12}
_LINEAR = {"spe1": 2, "ilu0": 20, "cpr": 5}


def work(case):
    if case["kind"] == "ensemble":
        n = sum(c["nx"] * c["ny"] * c["nz"] for c in _members(case))
    else:
        n = case["nx"] * case["ny"] * case["nz"]
    # per cell: an assembly reads the state and the static data and writes R and
    # the 7 blocks; a factorisation reads the blocks and writes 63 factor entries;
    # a BiCGStab iteration reads the blocks and the factors twice each and moves
    # about 30 vectors of three entries
    if case["kind"] == "products":
        return {"bytes": n * (2 * 504 + 4 * 24.0), "flops": n * (126.0 + 126.0)}
    spe1 = case.get("model") == "spe1"
    newton = case.get("iterations") or _NEWTON["spe1" if spe1 else case["kind"]]
    linear = newton * _LINEAR["spe1" if spe1 else case["precond"]]
    cpr = 900 if case["precond"] == "cpr" else 0
    return {"bytes": n * (newton * (100 + 528 + 504 + 504.0) + linear * (4 * 504 + 30 * 24 + 2 * cpr)),
            "flops": n * (newton * (1500 + 526.0) + linear * (4 * 126 + 60 + cpr / 4))}


# ---------------------------------------------------------------------------
# The same results from plain torch in 64 bits
# ---------------------------------------------------------------------------
class _Plain:
    """Residual of one implicit step (two-point fluxes, upwinding, reduced
    wells) as a differentiable function of the unknowns."""

    def __init__(self, m, state, dt):
        self.m, self.f, self.dt = m, m["fluid"], dt
        self.shape = (m["nz"], m["ny"], m["nx"])
        nz, ny, nx = self.shape
        t = lambda a: torch.as_tensor(a, device=DEV, dtype=F64)  # noqa: E731
        dx, dy, dz = t(m["dx"]), t(m["dy"]), t(m["dz"])
        k = t(m["perm"]).reshape(self.shape)
        ones = torch.ones(self.shape, device=DEV, dtype=F64)
        hx, hy, hz = ones * dx, ones * dy[:, None], ones * dz[:, None, None]
        self.pv = t(m["poro"]).reshape(self.shape) * hx * hy * hz
        self.depth = ones * (m["top_depth"] + torch.cumsum(dz, 0) - 0.5 * dz)[:, None, None]
        self.T = []
        for axis, (area, h) in ((2, (hy * hz, hx)), (1, (hx * hz, hy)), (0, (hx * hy, hz))):
            half = area * k / (0.5 * h)
            a, b = self._pair(half, axis)
            self.T.append((axis, a * b / (a + b)))
        self.flag = state[3].reshape(self.shape)
        self.wells = []
        q0 = self.cells(*(v.reshape(self.shape) for v in state[:3]), self.flag)
        self.acc0 = q0["acc"]
        for w in m["wells"]:
            ks = torch.tensor(w["ks"], device=DEV)
            at = (ks, torch.full_like(ks, w["j"]), torch.full_like(ks, w["i"]))
            ro = 0.14 * torch.sqrt(hx[at] ** 2 + hy[at] ** 2)
            wi = 2 * math.pi * k[at] * hz[at] / (torch.log(ro / w["rw"]) + w["skin"])
            a = {"water": 0, "gas": 2}[w["phase"]] if w["kind"] == "inj" else 1
            if w["kind"] == "inj":
                rho = q0["rho"][a][at][0]
            else:
                lam = [v[at] for v in q0["lam"]]
                rho = sum((l * r[at]).sum() for l, r in zip(lam, q0["rho"])) / sum(l.sum() for l in lam)
            head = self.f["g"] * rho * (self.depth[at] - self.depth[at][0])
            self.wells.append((w, at, wi, head, a))
        self.rate = [w["control"] == "rate" for w in m["wells"]]

    @staticmethod
    def _pair(v, axis):
        n = v.shape[axis]
        return v.narrow(axis, 0, n - 1), v.narrow(axis, 1, n - 1)

    def cells(self, p, sw, x, flag):
        f = self.f
        sat = flag == 0
        sg = torch.where(sat, x, torch.zeros_like(x))
        r = torch.where(sat, f["R_sb"] / f["p_b"] * p, x)
        so = 1 - sw - sg
        ps = f["p_b"] / f["R_sb"] * r
        b = [f["bw_ref"] * torch.exp(f["c_w"] * (p - f["p_ref"])),
             torch.exp(f["c_o"] * (p - ps)) / (1 + f["Bo_slope"] * r), p / (f["p_sc"] * f["Z"])]
        mu = [f["mu_w"], f["mu_o0"] / (1 + f["mu_o_r"] * r) * torch.exp(f["c_mu"] * (p - ps)),
              f["mu_g0"] * (1 + p / f["mu_g_p"])]
        rho = [f["rho_s"][0] * b[0], b[1] * (f["rho_s"][1] + f["rho_s"][2] * r), f["rho_s"][2] * b[2]]

        def corey(v):
            v = torch.where(v <= 0, torch.zeros_like(v), torch.where(v >= 1, torch.ones_like(v), v))
            return v ** f["n_corey"]

        dw, dg = 1 - f["s_wco"] - f["s_orw"], 1 - f["s_wco"] - f["s_org"]
        krow, krog = corey((so - f["s_orw"]) / dw), corey((so - f["s_org"]) / dg)
        ww = sw - f["s_wco"]
        ww = torch.where(ww < 0, torch.zeros_like(ww), ww)
        den = ww + sg
        low = den <= 1e-14
        kro = torch.where(low, krow, (ww * krow + sg * krog) / torch.where(low, torch.ones_like(den), den))
        lam = [corey((sw - f["s_wco"]) / dw) / mu[0], kro / mu[1], corey(sg / dg) / mu[2]]
        phi = torch.exp(f["c_r"] * (p - f["p_ref"]))
        acc = [phi * b[0] * sw, phi * b[1] * so, phi * (b[2] * sg + r * b[1] * so)]
        return {"b": b, "lam": lam, "rho": rho, "r": r, "acc": acc}

    def residual(self, p, sw, x, bhp, flag=None):
        """(R [3] over the cells, R_w per well) at the unknowns (cell arrays, bhp [nw])."""
        q = self.cells(p, sw, x, self.flag if flag is None else flag)
        R = [self.pv / self.dt * (a - a0) for a, a0 in zip(q["acc"], self.acc0)]
        mob = [b * l for b, l in zip(q["b"], q["lam"])]
        gas = q["r"] * mob[1]
        for axis, T in self.T:
            lo = [0] * 6
            hi = list(lo)
            hi[5 - 2 * axis], lo[4 - 2 * axis] = 1, 1     # pad behind / before along the axis
            back = lambda u: torch.nn.functional.pad(u, hi)  # noqa: E731
            front = lambda u: torch.nn.functional.pad(u, lo)  # noqa: E731
            zl, zh = self._pair(self.depth, axis)
            pl, ph = self._pair(p, axis)
            for a in range(3):
                rl, rh = self._pair(q["rho"][a], axis)
                d = (pl - ph) - self.f["g"] * 0.5 * (rl + rh) * (zl - zh)

                def flux(v):
                    vl, vh = self._pair(v, axis)
                    return torch.where(d >= 0, vl, vh) * T * d

                u = flux(mob[a])
                R[a] = R[a] + back(u) - front(u)
                if a == 1:
                    u = flux(gas)
                    R[2] = R[2] + back(u) - front(u)
        Rw = []
        for n, (w, at, wi, head, a) in enumerate(self.wells):
            d = p[at] - bhp[n] - head
            zero = torch.zeros_like(d)
            qs = [zero, zero, zero]
            if w["kind"] == "inj":
                lt = q["lam"][0][at] + q["lam"][1][at] + q["lam"][2][at]
                qs[a] = torch.where(d < 0, wi * lt * q["b"][a][at] * d, zero)
            else:
                for e in range(3):
                    qs[e] = torch.where(d > 0, wi * mob[e][at] * d, zero)
                qs[2] = qs[2] + torch.where(d > 0, wi * gas[at] * d, zero)
            R = [r.index_put(at, v, accumulate=True) for r, v in zip(R, qs)]
            total = -qs[a].sum() if w["kind"] == "inj" else qs[1].sum()
            Rw.append(total - w["target"] if self.rate[n] else bhp[n] - w["target"])
        return torch.stack([r.reshape(-1) for r in R]), torch.stack(Rw), qs

    def product(self, state, v):
        """The well-reduced operator at the state times v [n, 3]."""
        jvp = torch.func.jvp
        y = tuple(s.reshape(self.shape) for s in state[:3])
        u = tuple(v[:, e].reshape(self.shape) for e in range(3))
        fn = lambda p, sw, x, bhp: self.residual(p, sw, x, bhp)[:2]  # noqa: E731
        zero = tuple(torch.zeros_like(a) for a in y)
        bhp = state[4]
        _, (ax, bx) = jvp(fn, (*y, bhp), (*u, torch.zeros_like(bhp)))
        _, (_, d) = jvp(fn, (*y, bhp), (*zero, torch.ones_like(bhp)))
        _, (cx, _) = jvp(fn, (*y, bhp), (*zero, -bx / d))
        return (ax + cx).T.contiguous()

    def step(self, state, newton=40):
        """The converged implicit step: (p, sw, x, flag, bhp), or None."""
        f, n = self.f, state[0].numel()
        p, sw, x = (s.reshape(self.shape).clone() for s in state[:3])
        flag, bhp = self.flag.clone(), state[4].clone()
        for it in range(newton):
            def fn(v):
                c = v[:3 * n].reshape(3, *self.shape)
                R, Rw, _ = self.residual(c[0], c[1], c[2], v[3 * n:], flag)
                return torch.cat([R.reshape(-1), Rw])

            v = torch.cat([p.reshape(-1), sw.reshape(-1), x.reshape(-1), bhp])
            d = -torch.linalg.solve(torch.func.jacfwd(fn)(v), fn(v))
            dp, ds, dx = (a.reshape(self.shape) for a in d[:3 * n].reshape(3, n))
            size = max(float((dp / p).abs().max()), float(ds.abs().max()))
            sat = flag == 0
            dp = torch.maximum(torch.minimum(dp, 0.3 * p), -0.3 * p)
            top = torch.where(sat, torch.maximum(ds.abs(), dx.abs()), ds.abs())
            cut = torch.where(top > 0.2, 0.2 / top, torch.ones_like(top))
            ds = ds * cut
            dx = torch.where(sat, dx * cut, dx.clamp(-0.2 * f["R_sb"], 0.2 * f["R_sb"]))
            floor = 0.95 * f["p_b"] / f["R_sb"] * (x + dx)
            dp = torch.where(~sat & (p + dp < floor) & (floor < p), floor - p, dp)
            p, sw, x = p + dp, (sw + ds).clamp(0, 1), x + dx
            rs = f["R_sb"] / f["p_b"] * p
            x = torch.where(sat, torch.minimum(x, 1 - sw), x)
            gone, come = sat & (x < 0), ~sat & (x > rs * (1 + 1e-6))
            x = torch.where(gone, rs, torch.where(come, torch.zeros_like(x), x))
            flag = torch.where(gone, 1, torch.where(come, 0, flag.to(torch.int64))).to(torch.uint8)
            bhp = bhp + torch.maximum(torch.minimum(d[3 * n:], 0.3 * bhp), -0.3 * bhp)
            if size < 1e-13 and not bool((gone | come).any()):
                break
        else:
            return None
        if any(r and float(b) > w["bhp_limit"] for r, b, w in zip(self.rate, bhp, self.m["wells"])):
            return None
        return p, sw, x, flag, bhp

    def rates(self, p, sw, x, flag, bhp):
        """Surface rates [nw, 3] (production positive)."""
        out = []
        wells, rate = self.wells, self.rate
        for n in range(len(wells)):
            self.wells, self.rate = [wells[n]], [rate[n]]
            out.append(torch.stack([q.sum() for q in self.residual(p, sw, x, bhp[n:n + 1], flag)[2]]))
        self.wells, self.rate = wells, rate
        return torch.stack(out)


def exact(case, seed):
    """Products at any size, and the converged sub-step of small models; the
    linear algebra of larger steps (and a solve that stops at 1e-3) has none."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    if case["kind"] == "products":
        m = _model(case, g)
        state = _state(m, g)
        scale = torch.tensor([1e5, 0.05, 0.05], device=DEV, dtype=F64)
        v = torch.randn((m["nx"] * m["ny"] * m["nz"], 3), generator=g, device=DEV, dtype=F64) * scale
        return {"op": _Plain(m, state, case["days"] * DAY).product(state, v).reshape(-1), "prec": None}
    if case["kind"] == "step" and case["model"] == "spe1" and case["nx"] * case["ny"] * case["nz"] <= 2000:
        m = _model(case, g)
        state = _state(m, g)
        plain = _Plain(m, state, case["days"] * DAY)
        end = plain.step(state)
        if end is None:
            return None
        p, sw, x, flag, bhp = end
        return {"p": p.reshape(-1), "sw": sw.reshape(-1), "x": x.reshape(-1),
                "flag": None, "bhp": bhp, "rates": plain.rates(*end)}
    return None
