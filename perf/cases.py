"""Timing cases of the library: what a user's program has it do, and the same in plain 64-bit torch.

A case is one grid (or batch of grids) and a number of time steps between two
read-outs.  ``prepare`` builds the inputs and the contexts a program keeps,
``run`` is one pass through the public calls -- steps, then the fields (and
the sums, positions or gradients) the program came for -- and ``exact`` gives
what the first ``run`` returns, from a restatement of the method in float64.

Time-marching cases go on from pass to pass as a simulation does; cases with
``restart`` set their geometry at the start of each pass, as a parameter study
or an optimisation does for each evaluation.

Fields come back in the type of their context's arithmetic: float32 from FP32
and FP16-storage contexts, float64 from FP64 ones.  The pressure, the velocity
and the chemical potential of an FP16-storage context carry the resolution of
the 16-bit populations they are summed from and come back in 16 bits.  mdot,
the difference of two steps' liquid fractions, is returned by FP64 contexts.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2510_18688_gb300 import lbm, workloads as W

FLOW, PHASE, HEAT = W.FLOW, W.PHASE, W.HEAT


def listed():
    return [
        # The smallest grid (conduction freezing, Sec. 4.1): a few steps between
        # two looks at the ice front; launches and latency are what it costs.
        dict(name="column_400x4_fp32", kind="column", nx=400, ny=4, precision="fp32", steps=16),
        # The three-phase Stefan column (Sec. 4.2) in double precision, with the
        # conserved sums reduced during the steps, as a validation run takes them.
        dict(name="stefan_512x8_fp64", kind="stefan", nx=512, ny=8, precision="fp64", steps=64),
        # One point of a parameter study: a small droplet from its initial state,
        # its freezing curve (sums every 64 steps) and the fields at the end.
        dict(name="curve_160_fp32", kind="curve", nx=160, ny=160, precision="fp32", steps=256),
        # The headline workload (Sec. 4.3): 512 x 512, sums in every step.
        dict(name="droplet_512_fp32", kind="droplet", nx=512, ny=512, precision="fp32", steps=64),
        # The same in double precision: the reference of a convergence study.
        dict(name="droplet_512_fp64", kind="droplet", nx=512, ny=512, precision="fp64", steps=16),
        # The large grid (porous medium, Sec. 4.6): walls on all sides.
        dict(name="porous_2048x1024_fp32", kind="porous", nx=2048, ny=1024, precision="fp32", steps=16),
        # A large ragged grid with 16-bit population storage.
        dict(name="porous_1999x1001_fp16s", kind="porous", nx=1999, ny=1001, precision="fp16s", steps=16),
        # 64 droplets on cylinders of uneven sizes advanced together (Sec. 4.4).
        dict(name="batch_64_fp32", kind="batch", nx=512, ny=512, grids=64, precision="fp32", steps=8),
        # The rough fracture in three dimensions (Sec. 4.5).
        dict(name="fracture_256x128x30_fp32", kind="fracture", nx=256, ny=128, nz=30, precision="fp32", steps=8),
        # A smaller, ragged three-dimensional grid in double precision.
        dict(name="fracture_131x67x30_fp64", kind="fracture", nx=131, ny=67, nz=30, precision="fp64", steps=4),
        # Reverse mode: frozen fraction and its gradient with respect to every
        # parameter and to the initial temperature field.
        dict(name="gradient_256_fp64", kind="gradient", nx=256, ny=256, precision="fp64", steps=48),
        # Forward mode: fields and their derivatives along one parameter.
        dict(name="tangent_250x190", kind="tangent", nx=250, ny=190, precision="tangent", steps=8),
    ]


def draw(rng):
    def span(lo, hi):  # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["column", "stefan", "curve", "droplet", "droplet", "porous", "porous", "batch",
                       "fracture", "fracture", "gradient", "tangent"])
    if kind == "column":
        return dict(kind=kind, nx=span(128, 2048), ny=rng.randint(2, 12),
                    precision=rng.choice(["fp32", "fp64", "fp16s"]), steps=rng.randint(1, 40))
    if kind == "stefan":
        return dict(kind=kind, nx=span(128, 1024), ny=rng.randint(4, 24),
                    precision=rng.choice(["fp32", "fp64"]), steps=rng.randint(8, 64))
    if kind == "curve":
        n = span(64, 300)
        return dict(kind=kind, nx=n, ny=n, precision=rng.choice(["fp32", "fp64"]), steps=64 * rng.randint(1, 4))
    if kind == "droplet":
        return dict(kind=kind, nx=span(200, 1024), ny=span(200, 1024),
                    precision=rng.choice(["fp32", "fp32", "fp64", "fp16s"]), steps=rng.randint(4, 24))
    if kind == "porous":
        return dict(kind=kind, nx=span(600, 3000), ny=span(300, 2000),
                    precision=rng.choice(["fp32", "fp32", "fp16s"]), steps=rng.randint(2, 12))
    if kind == "batch":
        return dict(kind=kind, nx=512, ny=512, grids=span(3, 64), precision=rng.choice(["fp32", "fp32", "fp64"]),
                    steps=rng.randint(2, 8))
    if kind == "fracture":
        return dict(kind=kind, nx=span(48, 256), ny=span(40, 128), nz=rng.randint(16, 40),
                    precision=rng.choice(["fp32", "fp32", "fp64"]), steps=rng.randint(1, 6))
    if kind == "gradient":
        return dict(kind=kind, nx=span(96, 384), ny=span(96, 384), precision="fp64", steps=rng.randint(8, 48))
    return dict(kind=kind, nx=span(96, 512), ny=span(96, 512), precision="tangent", steps=rng.randint(2, 8))


# --- inputs -------------------------------------------------------------------


def _porous(nx, ny, seed):
    """The porous medium of ``workloads.porous`` (porosity 0.6, saturation 0.5)
    with its grains on a jittered lattice, built on the GPU."""
    r = W.rng(seed)
    x = torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5
    y = torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5

    def disks(cell, lo, hi, keep):
        best = torch.full((ny, nx), -1e3, dtype=torch.float64, device="cuda")
        for cy in np.arange(cell / 2, ny + cell / 2, cell):
            for cx in np.arange(cell / 2, nx + cell / 2, cell):
                rad, ox, oy, u = r.uniform(lo, hi), r.uniform(-1, 1), r.uniform(-1, 1), r.uniform()
                if u > keep:
                    continue
                px = cx + ox * max(0.0, cell / 2 - rad - 4.0)
                py = cy + oy * max(0.0, cell / 2 - rad - 4.0)
                i0, i1 = max(0, int(px - cell)), min(nx, int(px + cell))
                j0, j1 = max(0, int(py - cell)), min(ny, int(py + cell))
                if i0 < i1 and j0 < j1:
                    d = rad - torch.hypot(x[None, i0:i1] - px, y[j0:j1, None] - py)
                    best[j0:j1, i0:i1] = torch.maximum(best[j0:j1, i0:i1], d)
        return best

    eps = 4.0
    phi0 = 0.5 + 0.5 * torch.tanh(2.0 * disks(60.0, 15.0, 28.0, 0.9) / eps)
    phi = (1.0 - phi0) * torch.tanh(2.0 * disks(90.0, 30.0, 55.0, 0.75) / eps)
    p = W.base_params(nx, ny, cp_s=1.0, lambda_l=0.1, eps=eps, theta_deg=float(r.uniform(50.0, 70.0)),
                      latent=W.latent_from_stefan(float(r.uniform(0.1, 0.5))),
                      bc=("dirichlet", "dirichlet", "adiabatic", "adiabatic"),
                      T_wall=(-1.0, 0.1, 0.0, 0.0))
    p["lambda_s"] = 0.37
    return p, dict(phi0=phi0, phi=phi, T=torch.full_like(phi, 0.1), fl=torch.ones_like(phi))


def _one(case, seed):
    """(parameters, arrays) of a single grid."""
    kind, nx, ny = case["kind"], case["nx"], case["ny"]
    r = W.rng(1000 + seed)
    if kind == "column":
        return W.neumann(nx, ny, T0=float(r.uniform(0.0, 0.1)), ste=float(r.uniform(0.1, 0.5)),
                         alpha=float(r.uniform(0.1, 0.2)))
    if kind == "stefan":
        return W.stefan(nx, ny, hs=float(r.uniform(12.0, 20.0)), h0=float(r.uniform(0.15, 0.25)) * nx + 16.0,
                        ste=float(r.uniform(0.1, 0.3)))
    if kind == "porous":
        return _porous(nx, ny, seed)
    if kind == "fracture":
        return W.rough_fracture(nx, ny, case["nz"], seed=seed)
    return W.sessile_droplet(nx, seed=seed, radius=0.2 * min(nx, ny), ny=ny)


def _sides(case):
    return W.rng(case["grids"]).choice([128, 256, 384, 512], size=case["grids"])


def _grids(case, seed):
    if case["kind"] != "batch":
        return [_one(case, seed)]
    return [W.cylinder_droplet(int(n), seed=64 * seed + i) for i, n in enumerate(_sides(case))]


def _on_gpu(arrays):
    out = {k: torch.as_tensor(v, dtype=torch.float64, device="cuda").contiguous()
           for k, v in arrays.items() if k != "mask"}
    if arrays.get("mask") is not None:
        out["mask"] = torch.as_tensor(arrays["mask"], dtype=torch.uint8, device="cuda")
    return out


def _line(case):
    return (0, case["ny"] // 2)  # the row the ice front is followed along


def _direction(cfg):
    """d/dT of the cold substrate and wall (the latent heat held fixed)."""
    return {"T_wall": [0.0, 0.0, 1.0, 0.0], "T_cold": 1.0}


# --- one pass -----------------------------------------------------------------


def prepare(case, seed):
    kind, prec = case["kind"], case["precision"]
    three_d = kind == "fracture"
    diag_every = {"stefan": 8, "droplet": 1}.get(kind, 0)
    solvers, grids, nodes = [], [], []
    for cfg, arrays in _grids(case, seed):
        a = _on_gpu(arrays)
        if three_d:
            s = lbm.Solver3(cfg, precision=prec)
        else:
            s = lbm.Solver(cfg, precision=prec, diag_every=diag_every,
                           tangent=_direction(cfg) if prec == "tangent" else None)
        st = dict(solver=s, arrays=a, three_d=three_d)
        _set_geometry(st)
        torch.cuda.synchronize()
        solvers.append(s)
        grids.append(st)
        nodes.append(a["phi"].numel())
    names = lbm.FIELDS3 if three_d else lbm.FIELDS
    state = dict(case=case, grids=grids, solvers=solvers, nodes=nodes, names=names,
                 shape=(tuple(grids[0]["arrays"]["phi"].shape) if len(grids) == 1 else (sum(nodes),)))
    if kind == "batch":
        state["batch"] = lbm.Batch(solvers)
    return state


def _set_geometry(st):
    a = st["arrays"]
    mask = a["mask"].data_ptr() if "mask" in a else None
    f = lbm.lbm3_set_geometry if st["three_d"] else lbm.lbm_set_geometry
    f(st["solver"].ctx, a["phi0"].data_ptr(), mask, a["phi"].data_ptr(), a["T"].data_ptr(),
      a["fl"].data_ptr(), lbm.LBM_DEVICE, lbm._stream())


def _kept(names, prec):
    return [k for k in names if k != "mdot" or prec in ("fp64", "tangent")]


def _typed(v, names, kept, prec):
    """The planes of v by name, in the type of the context's arithmetic."""
    if prec in ("fp32", "fp16s"):
        v = v.float()
    out = {k: v[names.index(k)] for k in kept}
    if prec == "fp16s":
        out.update({k: out[k].bfloat16() for k in ("p", "ux", "uy", "mu")})
    return out


def _fields(state, tangent=False):
    """The fields of every grid, in device memory; a batch's one after another."""
    prec, names = state["case"]["precision"], state["names"]
    kept = _kept(names, prec)
    bits = sum(1 << names.index(k) for k in kept)
    out = torch.empty((len(names),) + state["shape"], dtype=torch.float64, device="cuda")
    flat = out.view(len(names), -1)
    at = 0
    for st, n in zip(state["grids"], state["nodes"]):
        ptrs = [flat[i, at:].data_ptr() if k in kept else None for i, k in enumerate(names)]
        if st["three_d"]:
            read = lbm.lbm3_read_fields
        else:
            read = lbm.lbm_read_tangent_fields if tangent else lbm.lbm_read_fields
        read(st["solver"].ctx, bits, ptrs, lbm.LBM_DEVICE, lbm._stream())
        at += n
    return _typed(out, names, kept, prec)


SUMS = ("mass", "material_mass", "rhoH", "liquid_volume", "material_volume", "frozen_volume",
        "phi_sum", "kinetic")


def _sums(d, prec):
    return np.array([d[k] for k in SUMS], dtype=np.float64 if prec == "fp64" else np.float32)


def run(state):
    case = state["case"]
    kind, n, prec = case["kind"], case["steps"], case["precision"]
    s = state["solvers"][0]
    out = {}
    if kind in ("curve", "gradient"):
        _set_geometry(state["grids"][0])
    if kind == "gradient":
        value, grad, dT0 = s.adjoint_coupled(n, observable=0, every=16, initial_T=True)
        return dict(value=value, grad=np.array(grad), dT0=dT0, **_fields(state))
    if kind == "batch":
        state["batch"].step(n)
        return _fields(state)
    if kind == "curve":
        curve = []
        for _ in range(n // 64):
            s.step(64)
            curve.append(_sums(s.diagnostics(), prec))
        out["curve"] = np.stack(curve)
    else:
        s.step(n)
    if kind in ("stefan", "droplet") and prec != "fp16s":
        out["sums"] = _sums(s.diagnostics(compute=False), prec)
    if kind == "column":
        out["front"] = np.array(s.crossings(*_line(case))[1],
                                dtype=np.float64 if prec == "fp64" else np.float32)
    out.update(_fields(state))
    if kind == "tangent":
        out["derivatives"] = _fields(state, tangent=True)
    return out


def work(case):
    """Per node and step: the populations and lagged fields read and written
    once, the static fields read; the arithmetic of the local state, the
    stencils and the three collisions.  Then the fields, written once."""
    kind, prec = case["kind"], case["precision"]
    if kind == "batch":
        nodes = int((_sides(case) ** 2).sum())
    else:
        nodes = case["nx"] * case["ny"] * case.get("nz", 1)
    pops, lags, flops, fields = (57, 7, 1500, 13) if kind == "fracture" else (27, 6, 700, 12)
    if kind == "column":
        pops, flops = 18, 350
    real = {"fp64": 8, "tangent": 16}.get(prec, 4)
    pop = 2 if prec == "fp16s" else real
    if kind != "fracture" and prec in ("fp32", "fp16s"):
        lags = 7
    step = 2 * pops * pop + 2 * lags * real + real + 1
    back = fields * (16 if prec == "tangent" else 8)
    if prec == "tangent":
        flops *= 3
    steps = case["steps"]
    if kind == "gradient":  # forward, recomputed, and reversed with the adjoint state in and out
        return dict(bytes=nodes * (steps * (3.5 * step) + back), flops=nodes * steps * 4.0 * flops)
    return dict(bytes=nodes * (steps * step + back), flops=nodes * steps * float(flops))


# --- the method in 64 bits ------------------------------------------------------
#
# Plain torch, float64, one tensor per population; D2Q9 or D3Q19 by the number of
# axes.  Axis order of tensors is [z,] y, x; vectors are (x, y[, z]).


def _lattice(dim):
    axes = [tuple(s if k == a else 0 for k in range(dim)) for a in range(dim) for s in (1, -1)]
    diag = [tuple(s if k == a else t if k == b else 0 for k in range(dim))
            for a in range(dim) for b in range(a + 1, dim) for s in (1, -1) for t in (1, -1)]
    w0, wa, wd = (4 / 9, 1 / 9, 1 / 36) if dim == 2 else (1 / 3, 1 / 18, 1 / 36)
    c = [(0,) * dim] + axes + diag
    w = [w0] + [wa] * len(axes) + [wd] * len(diag)
    return c, w, [c.index(tuple(-v for v in e)) for e in c]


class _Plain:
    """The coupled step on one grid.  `over` replaces scalars of the parameter set
    by tensors (for derivatives)."""

    def __init__(self, cfg, arrays, over=None):
        g = dict(cfg, **(over or {}))
        self.dim = 3 if "nz" in cfg else 2
        self.c, self.w, self.opp = _lattice(self.dim)
        self.bc = cfg["bc"]
        self.lat = cfg["lattices"]
        self.Tw = g["T_wall"]
        self.g = g
        self.force = [g["gx"], g["gy"]] + ([g["gz"]] if self.dim == 3 else [])
        self.phi0 = arrays["phi0"]
        self.mask = arrays["mask"] != 0 if "mask" in arrays else None
        cps, cpl = g["cp_s"], g["cp_l"]
        self.rr = g["rho_ref"] * 2 * cps * cpl / (cps + cpl)
        deg = math.pi / 180

        def cos(v):
            return torch.cos(v * deg) if torch.is_tensor(v) else math.cos(v * deg)

        self.ct, self.cp = cos(g["theta_deg"]), cos(g["psi_deg"])
        self.itg = 1 / (0.5 + 3 * g["mobility"] / g["eta"])
        # links that leave through a wall: the first axis crossed decides
        shape = self.phi0.shape
        pos = [torch.arange(n, device="cuda").view([-1 if k == i else 1 for k in range(self.dim)])
               for i, n in enumerate(shape)]
        self.cross = []
        for e in self.c:
            hit, here = [], torch.zeros(shape, dtype=torch.bool, device="cuda")
            for a in range(self.dim):
                ax = self.dim - 1 - a
                if e[a] == 0 or self.bc[2 * a] == "periodic":
                    continue
                side = 2 * a + (1 if e[a] > 0 else 0)
                at = (pos[ax] == (shape[ax] - 1 if e[a] > 0 else 0)).expand(shape) & ~here
                hit.append((side, at))
                here = here | at
            self.cross.append(hit)

    def mix(self, fs, w, name):
        g = self.g
        return fs * g[name + "_s"] + (1 - fs) * (w * g[name + "_l"] + (1 - w) * g[name + "_g"])

    def cap(self, fs, w):
        return self.mix(fs, w, "rho") * self.mix(fs, w, "cp")

    def at(self, v, e):
        """v(x + e), the wall node mirrored beyond a wall."""
        for a in range(self.dim):
            if e[a] == 0:
                continue
            ax = self.dim - 1 - a
            if self.bc[2 * a] == "periodic":
                v = torch.roll(v, -e[a], ax)
            else:
                n = v.shape[ax]
                edge = v.narrow(ax, n - 1 if e[a] > 0 else 0, 1)
                part = v.narrow(ax, 1 if e[a] > 0 else 0, n - 1)
                v = torch.cat([part, edge] if e[a] > 0 else [edge, part], ax)
        return v

    def grad(self, v):
        out = [0.0] * self.dim
        for e, w in zip(self.c[1:], self.w[1:]):
            n = self.at(v, e)
            for a in range(self.dim):
                if e[a]:
                    out[a] = out[a] + 3 * w * e[a] * n
        return out

    def lap(self, v):
        return sum(6 * w * (self.at(v, e) - v) for e, w in zip(self.c[1:], self.w[1:]))

    def chem(self, phi, fs):
        g, q = self.g, self.phi0
        a = 3 * g["sigma"] / g["eps"]
        return (a * phi * (phi - 1) * (phi + 1) + 3 * a * q * q * phi
                + a * self.ct * q * (3 * phi * phi + q * q - 1) + 3 * a * fs * fs * phi
                + a * self.cp * fs * (3 * phi * phi + fs * fs - 1)
                - 3 * g["eps"] * g["sigma"] / 8 * (self.lap(phi) + self.ct * self.lap(q) + self.cp * self.lap(fs)))

    def start(self, phi, T, fl):
        q = self.phi0
        zero = torch.zeros_like(q)
        w = ((1 - q + phi) / 2).clamp(0, 1)
        fl = fl.clamp(0, 1)
        fs = q + w * (1 - fl)
        fs = torch.where(fs > 1, 1.0, fs)
        emu = self.g["eta"] * self.chem(phi, fs)
        fsf = torch.where(q + w > 1, 1.0, q + w)
        rhoH = torch.where(T < 0, self.cap(fsf, w), self.cap(q, w)) * T + w * self.g["rho_l"] * self.g["latent"] * fl
        f = [zero for _ in self.c]
        gg = [phi + (self.w[0] - 1) * emu] + [v * emu for v in self.w[1:]]
        h = [rhoH - (1 - self.w[0]) * self.rr * T] + [v * self.rr * T for v in self.w[1:]]
        return f, gg, h, (fl, w, zero, [zero] * self.dim, zero)

    def macros(self, state):
        f, gg, h, (flp, wp, pp, _, Qp) = state
        g, q = self.g, self.phi0
        zero = torch.zeros_like(q)
        m = {}
        ell = wp * g["rho_l"] * g["latent"]
        fsf = torch.where(q + wp > 1, 1.0, q + wp)
        if self.mask is not None and self.lat & HEAT:
            Tc = g["T_cold"]
            cold = float(Tc) < 0
            r = (self.cap(fsf, wp) if cold else self.cap(q, wp)) * Tc + (0.0 if cold else ell)
            h = [torch.where(self.mask, (r - (1 - self.w[0]) * self.rr * Tc) if i == 0 else self.w[i] * self.rr * Tc, v)
                 for i, v in enumerate(h)]
        T, fl, rhoH, mdot = zero, flp, zero, zero
        if self.lat & HEAT:
            rhoH = sum(h) + Qp / 2
            low, high = rhoH < 0, rhoH > ell
            T = torch.where(low, rhoH / self.cap(fsf, wp), torch.where(high, (rhoH - ell) / self.cap(q, wp), 0.0))
            some = torch.where(ell > 0, ell, 1.0)
            fl = torch.where(low, 0.0, torch.where(high, 1.0, torch.where(ell > 0, rhoH / some, 1.0)))
            mdot = (1 - g["rho_s"] / g["rho_l"]) * wp * (flp - fl)
        if self.lat & PHASE:
            phi = sum(gg) / (1 - mdot / 2)
            w = ((1 - q + phi) / 2).clamp(0, 1)
        else:
            w, phi = wp, 2 * wp - 1 + q
        fs = q + w * (1 - fl)
        fs = torch.where(fs > 1, 1.0, fs)
        rho = self.mix(fs, w, "rho")
        mu, F = zero, [rho * v for v in self.force]
        if self.lat & PHASE:
            mu = self.chem(phi, fs)
            F = [a + mu * b for a, b in zip(F, self.grad(phi))]
        u, p, S, Ft, G, tauf = [zero] * self.dim, zero, zero, F, F, None
        if self.lat & FLOW:
            gr, gp = self.grad(rho), self.grad(pp)
            us = [(sum(e[a] * v for e, v in zip(self.c, f) if e[a]) + F[a] / 2) / rho for a in range(self.dim)]
            u = [v - fs * v / 2 for v in us]
            S = rho * mdot + sum(a * b for a, b in zip(u, gr))
            Ft = [a - (b - c / 3) for a, b, c in zip(F, gp, gr)]
            G = [a - rho * fs * b for a, b in zip(F, us)]
            uFt = sum(a * b for a, b in zip(u, Ft))
            uu = sum(a * a for a in u)
            tauf = 3 * self.mix(fs, w, "mu") / rho + 0.5
            p = (sum(f[1:]) + S / 2 + (tauf - 0.5) * self.w[0] * (S - 3 * uFt)
                 - 1.5 * rho * self.w[0] * uu) / (3 * (1 - self.w[0]))
        m.update(phi=phi, fs=fs, fl=fl, T=T, rhoH=rhoH, p=p, u=u, rho=rho, mu=mu, w=w, mdot=mdot,
                 S=S, Ft=Ft, G=G, tauf=tauf, h=h)
        return m

    def step(self, state):
        f, gg, _, (_, _, _, phup, _) = state
        g, m = self.g, self.macros(state)
        h, u, phi, rho, mdot, fs, w, T = (m[k] for k in ("h", "u", "phi", "rho", "mdot", "fs", "w", "T"))
        uu = sum(a * a for a in u)

        def dot(e, v):
            return sum(a * b for a, b in zip(e, v) if a) if any(e) else 0.0

        nf, ng, nh = f, gg, h
        C = rho * self.mix(fs, w, "cp")
        if self.lat & FLOW:
            it = 1 / m["tauf"]
            k = 1 - it / 2
            uFt = dot([1] * self.dim, [a * b for a, b in zip(u, m["Ft"])])
            nf = []
            for i, e in enumerate(self.c):
                cu = dot(e, u)
                eq = (3 * (self.w[i] - (i == 0)) * m["p"]
                      + self.w[i] * rho * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
                src = self.w[i] * (m["S"] - 3 * uFt + 3 * dot(e, m["G"]) + 9 * cu * dot(e, m["Ft"]))
                nf.append(f[i] * (1 - it) + it * eq + k * src)
            nf = self.stream(nf, False)
        phu = [phi * v for v in u]
        if self.lat & PHASE:
            k = 1 - self.itg / 2
            emu = g["eta"] * m["mu"]
            V = [3 * (self.itg * a + k * (a - b)) for a, b in zip(phu, phup)]
            ng = []
            for i, e in enumerate(self.c):
                eq = phi + (self.w[0] - 1) * emu if i == 0 else self.w[i] * emu
                ng.append(gg[i] * (1 - self.itg) + self.itg * eq + self.w[i] * (k * phi * mdot + dot(e, V)))
            ng = self.stream(ng, False)
        if self.lat & HEAT:
            ia = 1 / (0.5 + 3 * self.mix(fs, w, "lambda") / self.rr)
            CT = C * T
            nh = []
            for i, e in enumerate(self.c):
                o = self.opp[i]
                cu = dot(e, u)
                rest = m["rhoH"] - self.rr * T if i == 0 else 0.0
                es = rest + self.w[i] * (self.rr * T + CT * (4.5 * cu * cu - 1.5 * uu))
                ea = self.w[i] * CT * 3 * cu
                nh.append(h[i] - (2 - ia) * ((h[i] + h[o]) / 2 - es) - ia * ((h[i] - h[o]) / 2 - ea)
                          + (1 - ia / 2) * self.w[i] * CT * mdot)
            nh = self.stream(nh, True)
        zero = torch.zeros_like(phi)
        lag = (m["fl"], w, m["p"], phu if self.lat & PHASE else [zero] * self.dim,
               C * T * mdot if self.lat & HEAT else zero)
        return nf, ng, nh, lag

    def stream(self, post, heat):
        out = []
        for i, e in enumerate(self.c):
            v = torch.roll(post[i], [e[a] for a in range(self.dim)], [self.dim - 1 - a for a in range(self.dim)])
            o = self.opp[i]  # population i of a node that sent o through a wall comes back there
            for side, where in self.cross[o]:
                back = post[o]
                if heat and self.bc[side] == "dirichlet":
                    back = -back + 2 * self.w[i] * self.rr * self.Tw[side]
                v = torch.where(where, back, v)
            out.append(v)
        return out

    def fields(self, state):
        m = self.macros(state)
        out = {k: m[k] for k in ("phi", "fs", "fl", "T", "rhoH", "p", "rho", "mu", "w", "mdot")}
        out.update(zip(("ux", "uy", "uz"), m["u"]))
        return out

    def sums(self, state):
        g, m = self.g, self.macros(state)
        w, fl = m["w"], m["fl"]
        uu = sum(a * a for a in m["u"])
        v = [m["rho"], w * (g["rho_s"] * (1 - fl) + g["rho_l"] * fl), m["rhoH"], w * fl, w, w * (1 - fl),
             m["phi"], m["rho"] * uu / 2]
        return np.array([float(x.sum()) for x in v])


def _crossing(s, level=0.5):
    """The last crossing of `level` along a line of values (NaN if none)."""
    d = (s - level).cpu().numpy()
    k = np.nonzero((d[:-1] <= 0) != (d[1:] <= 0))[0]
    return np.array(k[-1] + d[k[-1]] / (d[k[-1]] - d[k[-1] + 1]) if len(k) else np.nan)


def _exact_gradient(case, cfg, a):
    names = ("T_wall", "latent", "theta_deg", "sigma", "gx", "gy", "T_cold")
    over = {k: torch.tensor(cfg[k], dtype=torch.float64, device="cuda", requires_grad=True) for k in names}
    T0 = a["T"].clone().requires_grad_(True)
    P = _Plain(cfg, a, over)
    state = P.start(a["phi"], T0, a["fl"])
    for _ in range(case["steps"]):
        state = torch.utils.checkpoint.checkpoint(P.step, state, use_reentrant=False)
    m = P.macros(state)
    value = (m["w"] * (1 - m["fl"])).sum() / m["w"].sum()
    got = torch.autograd.grad(value, [over[k] for k in names] + [T0], allow_unused=True)
    got = [torch.zeros_like(v) if d is None else d for d, v in zip(got, [over[k] for k in names] + [T0])]
    grad = torch.cat([v.reshape(-1) for v in got[:-1]]).cpu().numpy()
    with torch.no_grad():
        out = {k: v.detach() for k, v in P.fields(state).items()}
    return dict(value=float(value.detach()), grad=grad, dT0=got[-1].cpu().numpy(), **out)


def _exact_tangent(case, cfg, a):
    import torch.autograd.forward_ad as fwd
    d = _direction(cfg)
    with fwd.dual_level():
        one = torch.ones((), dtype=torch.float64, device="cuda")

        def dual(v, t):
            return fwd.make_dual(one * v, one * t)

        over = dict(T_wall=[dual(v, t) for v, t in zip(cfg["T_wall"], d["T_wall"])],
                    T_cold=dual(cfg["T_cold"], d["T_cold"]))
        P = _Plain(cfg, a, over)
        state = P.start(a["phi"], a["T"], a["fl"])
        for _ in range(case["steps"]):
            state = P.step(state)
        out, der = {}, {}
        for k, v in P.fields(state).items():
            x, t = fwd.unpack_dual(v)
            out[k] = x.clone()
            der[k] = torch.zeros_like(x) if t is None else t.clone()
    return dict(out, derivatives=der)


def exact(case, seed):
    kind, prec, n = case["kind"], case["precision"], case["steps"]
    grids = [(cfg, _on_gpu(arrays)) for cfg, arrays in _grids(case, seed)]
    cfg, a = grids[0]
    if kind == "gradient":
        return _exact_gradient(case, cfg, a)
    if kind == "tangent":
        return _exact_tangent(case, cfg, a)
    parts, out = [], {}
    with torch.no_grad():
        for cfg, a in grids:
            P = _Plain(cfg, a)
            state = P.start(a["phi"], a["T"], a["fl"])
            curve = []
            for k in range(n):
                if kind in ("stefan", "droplet") and prec != "fp16s":
                    every = 8 if kind == "stefan" else 1
                    if k == (n - 1) - (n - 1) % every:
                        out["sums"] = P.sums(state)
                state = P.step(state)
                if kind == "curve" and (k + 1) % 64 == 0:
                    curve.append(P.sums(state))
            if curve:
                out["curve"] = np.stack(curve)
            fields = P.fields(state)
            if kind == "column":
                axis, row = _line(case)
                out["front"] = _crossing((fields["w"] * (1 - fields["fl"]))[row])
            parts.append(fields)
    for k in _kept(lbm.FIELDS3 if kind == "fracture" else lbm.FIELDS, prec):
        out[k] = parts[0][k] if len(parts) == 1 else torch.cat([p[k].reshape(-1) for p in parts])
    return out
