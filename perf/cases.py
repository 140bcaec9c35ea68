"""What this library is timed on: whole parameter-study passes through its public entry points.

A pass is what a study of the paper's cases does once its lattices exist: put an initial state in
(densities of every case), take a number of time steps, and read the fields back, with the
diagnostics and contact angles where the study reads them.  Real runs take thousands of steps
between two reads; the passes here take 16 to 100 so that they stay short.

Fields leave the library as FP64 arrays whatever the storage mode.  A pass hands them on in the
precision the mode computes or stores them in (FP64, FP32, FP16 or BF16), as one [fields][nodes]
block: densities and velocities in lattice units side by side.

``exact`` is the same pass in plain torch, FP64 throughout, written from the model's equations.
"""
import itertools
import math

import numpy as np
import torch

from paper_2505_22256_gb300 import lbm, lbm3d
from paper_2505_22256_gb300 import scenarios as S

OUT_TYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
ELEM = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}


# ------------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------------
def _case(kind, storage, steps, nx, ny, nz=1, ncases=1, read="fields", host=False, reading="e8", name=None):
    c = {"kind": kind, "storage": storage, "steps": steps, "nx": nx, "ny": ny, "nz": nz, "ncases": ncases,
         "read": read, "host": host, "reading": reading}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: the plain FP64 form of the cylinder case, one 96 x 96 lattice, fields to the host
        _case("cylinder", "f64", 50, 96, 96, host=True, name="cylinder96_f64"),
        # two-layer Couette flow between sliding walls at the paper's 50 x 100, three wall angles, read
        # to the host with the diagnostics as the co-current study does
        _case("couette", "f32", 100, 50, 100, ncases=3, read="diagnostics", host=True, name="couette3_f32"),
        # a droplet driven past a square obstacle: one 350 x 150 channel with inlet and outflow
        _case("obstacle", "f32", 100, 350, 150, name="obstacle_f32"),
        # both adhesion schemes at seven angles on the paper's 300 x 350 box (periodic both ways), with
        # diagnostics and contact angles: the scheme study
        _case("box", "f32", 50, 300, 350, ncases=14, read="all", name="schemes14_f32"),
        # droplet through a throat, 2048 x 512, FP16 shifted storage
        _case("throat", "f16", 50, 2048, 512, name="throat_f16"),
        # the headline sweep: seven 1024 x 1024 cylinder cases, FP32, and its FP16 storage form
        _case("cylinder", "f32", 32, 1024, 1024, ncases=7, name="sweep7_f32"),
        _case("cylinder", "f16", 32, 1024, 1024, ncases=7, name="sweep7_f16"),
        # immiscible displacement through the 4096 x 2048 porous medium (open x, 40 % solid)
        _case("porous", "f32", 20, 4096, 2048, name="porous_f32"),
        # a batch of uneven contact-angle cases, sides 64..512, flat and cylindrical walls, monitored
        _case("ensemble", "f32", 32, 512, 512, ncases=64, read="all", name="ensemble64_f32"),
        # 3-D droplet on a sphere: a small lattice read with diagnostics and contact angle, the
        # paper's 200 x 200 x 280 in FP32, and a half-scale one in FP16 storage
        _case("sphere", "f32", 50, 40, 40, 56, read="all", name="sphere40_f32"),
        _case("sphere", "f32", 16, 200, 200, 280, read="all", name="sphere200_f32"),
        _case("sphere", "f16", 32, 100, 100, 140, name="sphere100_f16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cylinder", "cylinder", "couette", "obstacle", "box", "throat", "porous", "ensemble", "sphere",
                       "sphere"])
    storage = rng.choice(["f32", "f32", "f32", "f16", "f16", "bf16"])
    reading = rng.choice(["e8", "e8", "e8", "psi", "first"])
    read = rng.choice(["fields", "all"]) if storage == "f32" and kind in ("cylinder", "box", "ensemble", "sphere") else "fields"
    steps = rng.randint(16, 40)
    if kind == "cylinder":
        n = _log(rng, 96, 1024)
        if n <= 128 and rng.random() < 0.5:
            storage, read = "f64", "fields"
        return _case(kind, storage, steps, n, n, ncases=rng.randint(1, 7), read=read, reading=reading)
    if kind == "couette":
        return _case(kind, storage, steps, rng.randint(48, 160), rng.randint(64, 200), ncases=_log(rng, 1, 64),
                     reading=reading)
    if kind == "obstacle":
        nx = _log(rng, 300, 1200)
        return _case(kind, storage, steps, nx, int(nx * rng.uniform(0.4, 0.5)), ncases=rng.randint(1, 3), reading=reading)
    if kind == "box":
        nx = rng.randint(280, 420)
        return _case(kind, storage, steps, nx, nx + rng.randint(40, 70), ncases=rng.randint(1, 14), read=read,
                     reading=reading)
    if kind == "throat":
        nx = _log(rng, 512, 2048)
        return _case(kind, storage, steps, nx, nx // 4 + rng.randint(0, 9), reading=reading)
    if kind == "porous":
        nx = _log(rng, 1024, 4096)
        return _case(kind, storage, 20, nx, nx // 2 - rng.randint(0, 9), reading=reading)
    if kind == "ensemble":
        n = _log(rng, 128, 512)
        return _case(kind, storage, steps, n, n, ncases=_log(rng, 4, 64), read=read, reading=reading)
    n = _log(rng, 32, 190)
    return _case(kind, storage, 16, n, n + rng.randint(0, 9), int(1.4 * n), read=read, reading=reading)


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _scenarios(case, seed):
    """The seeded scenario objects of a case (masks, initial densities, parameters)."""
    kind, nx, ny, n = case["kind"], case["nx"], case["ny"], case["ncases"]
    angles = [30.0 + 120.0 * (k + 0.5) / n for k in range(n)]
    seed = int(seed) % (1 << 22)
    if kind == "cylinder":
        out = [S.cylinder_droplet(nx, R=160.0 * nx / 1024.0, r=200.0 * nx / 1024.0, lam=S.lambda_for_angle(t),
                                  seed=seed + k) for k, t in enumerate(angles)]
    elif kind == "couette":
        out = [S.couette_channel(nx, ny, lam=S.lambda_for_angle(t), seed=seed + k) for k, t in enumerate(angles)]
    elif kind == "obstacle":
        f = ny / 150.0
        out = [S.square_obstacle_channel(nx, ny, int(25 * f), (int(122 * f), int(75 * f)), 25 * f,
                                         (int(55 * f), int(75 * f)), theta=t, seed=seed + k)
               for k, t in enumerate(angles)]
    elif kind == "box":
        f = nx / 300.0
        out = [S.cylinder_in_box(nx, ny, 70 * f, (nx / 2, 130 * f), 50 * f, (nx / 2, 230 * f),
                                 lam=S.lambda_for_angle(angles[k - k % 2]), seed=seed + k,
                                 scheme=("improved", "original")[k % 2]) for k in range(n)]
    elif kind == "throat":
        f = nx / 2048.0
        out = [S.throat_channel(nx, ny, 180.0 * f, 120.0 * f, seed=seed)]
    elif kind == "porous":
        out = [S.porous_disks(nx, ny, seed=seed)]
    elif kind == "ensemble":
        sides, lams = np.random.default_rng(1000 * nx + n).integers(64, nx + 1, n), np.random.default_rng(seed)
        out = [S.flat_droplet(m, m, m / 5.0, S.lambda_for_angle(lams.uniform(30, 150)), seed + k) if k % 2 else
               S.cylinder_droplet(m, m / 6.0, m / 5.0, S.lambda_for_angle(lams.uniform(30, 150)), seed + k)
               for k, m in enumerate(int(m) for m in sides)]
    else:
        k = nx / 200.0
        out = [S.sphere_droplet_3d(nx, ny, case["nz"], 50 * k, (100 * k, 100 * k, 100 * k), 45 * k,
                                   (100 * k, 100 * k, 180 * k), seed=seed)]
    for sc in out:
        if case["reading"] == "psi":
            sc.second_layer = "psi"
        elif case["reading"] == "first":
            sc.adhesion_stencil = "d3q19" if kind == "sphere" else "d2q9"
    return out


_program = {}  # the one side stream that a program runs its lattices on


def prepare(case, seed):
    """The lattice handle(s) of a case on the program's stream, the initial densities on the device, and
    the array the fields are written to."""
    scs = _scenarios(case, seed)
    if "stream" not in _program:
        _program["stream"] = torch.cuda.Stream()
    st = {"case": case, "stream": _program["stream"], "surfaces": None}
    handle = st["stream"].cuda_stream
    if case["kind"] == "sphere":
        sc = scs[0]
        st["lat"] = lbm3d.Lattice3(sc.solid, sc.rhoA0, sc.rhoB0, sc.params(), case["storage"], handle)
        st["surfaces"] = sc.sphere
    else:
        st["lat"] = lbm.Lattice(scs, case["storage"], handle)
        st["surfaces"] = [sc.surface for sc in scs]
    for k, key in enumerate(("rhoA0", "rhoB0")):
        st["AB"[k]] = torch.from_numpy(np.concatenate([getattr(sc, key).reshape(-1) for sc in scs])).cuda()
    st["out"] = torch.zeros(5 if case["kind"] == "sphere" else 4, st["A"].numel(), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return st


def _numbers(rows, dtype):
    return torch.tensor(rows, dtype=torch.float64).to(dtype)


DIAG2 = ("mass_A", "mass_B", "mom_x", "mom_y", "umax", "rhoA_min", "rhoA_max", "rhoB_min", "rhoB_max")
DIAG3 = DIAG2[:4] + ("mom_z",) + DIAG2[4:]


# ------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------
def run(st):
    case, lat = st["case"], st["lat"]
    dtype = OUT_TYPE[case["storage"]]
    res = {}
    with torch.cuda.stream(st["stream"]):
        out = st["out"]
        if case["kind"] == "sphere":
            lat.set_densities(st["A"], st["B"], on_device=True)
            lat.step(case["steps"])
            if case["read"] == "all":
                res["angle"] = _numbers(lat.contact_angle(st["surfaces"])[:2], dtype)
                d = lat.diagnostics(allow_unstable=True)
                res["diag"], res["n_fluid"] = _numbers([d[k] for k in DIAG3], dtype), d["n_fluid"]
            status = lbm.load_library().lbm3d_fields(lat.ctx, *[o.data_ptr() for o in out], 1)
            assert status == lbm.LBM_OK
            res["fields"] = out.to(dtype)
            return res
        lbm.lbm_set_densities_all(lat.ctx, st["A"], st["B"], on_device=True)
        lat.step(case["steps"])
        if case["read"] in ("all", "diagnostics"):
            d = lat.diagnostics_all(allow_unstable=True)
            res["diag"] = _numbers([[x[k] for k in DIAG2] for x in d], dtype)
            res["n_fluid"] = torch.tensor([x["n_fluid"] for x in d])
        if case["read"] == "all":
            theta, rms, _ = lat.contact_angle_all(st["surfaces"])
            res["angle"] = _numbers(np.stack([theta, rms]).tolist(), dtype)
        if case["host"]:
            f = lat.fields_all()
            res["fields"] = torch.from_numpy(np.stack([np.concatenate([x[q].reshape(-1) for x in f]) for q in range(4)])).to(dtype)
        else:
            lbm.lbm_fields_all(lat.ctx, *out, on_device=True)
            res["fields"] = out.to(dtype)
    return res


def work(case):
    """State in and out once per step and fluid node; densities in, fields out."""
    q, per = (19, 1400) if case["kind"] == "sphere" else (9, 420)
    nodes = case["nx"] * case["ny"] * case["nz"] * case["ncases"]
    if case["kind"] == "ensemble":
        nodes = case["ncases"] * (case["nx"] ** 2 + 64 * case["nx"] + 64 ** 2) / 3.0  # sides uniform in 64..nx
    fluid = nodes * {"porous": 0.6, "box": 0.85, "cylinder": 0.96, "throat": 0.90, "ensemble": 0.95, "sphere": 0.953,
                     "obstacle": 0.988, "couette": 1.0}[case["kind"]]
    state = 2 * q * ELEM[case["storage"]] * fluid
    fields = 8 * (5 if case["kind"] == "sphere" else 4) * nodes
    return {"bytes": 2.0 * state * case["steps"] + 16.0 * nodes + state + fields, "flops": per * fluid * case["steps"]}


# ------------------------------------------------------------------------------------------------
# the same pass in 64 bits: arrays [y, x] or [z, y, x], offsets (ex, ey[, ez])
# ------------------------------------------------------------------------------------------------
E2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
E3 = [e for e in itertools.product((0, 1, -1), repeat=3) if sum(abs(v) for v in e) <= 2]
W2 = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
W3 = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
G2 = {1: 4 / 21, 2: 4 / 45, 4: 1 / 60, 5: 2 / 315, 8: 1 / 5040}
G3 = {1: 4 / 45, 2: 1 / 21, 3: 2 / 105, 4: 5 / 504, 5: 1 / 315, 6: 1 / 630, 8: 1 / 5040}


def _sq(e):
    return sum(v * v for v in e)


def _sgn(e):
    return tuple((v > 0) - (v < 0) for v in e)


class _Exact:
    def __init__(self, sc, dev):
        self.sc, self.dev = sc, dev
        solid = torch.from_numpy(sc.solid.astype(bool)).to(dev)
        self.d = d = solid.dim()
        self.E, self.W, self.G = (E2, W2, G2) if d == 2 else (E3, W3, G3)
        self.opp = [self.E.index(tuple(-v for v in e)) for e in self.E]
        self.bc = [getattr(sc, "bc_x", "periodic"), getattr(sc, "bc_y", "periodic"), "periodic"][:d]  # x, y, z
        self.solid, self.fluid = solid, ~solid
        self.solid1 = self.pad(solid, True, clamp=True)      # first layer: beyond an open column is that column
        self.nofluid = self.pad(solid, True, clamp=False)    # second layer: outside a wall or an open column
        p = sc.params()
        self.tau, self.Gc, self.lam, self.delta = p["tau"], p["G"], p["lam"], p["delta"]
        self.Gw2 = p["G"] if p["Gw2"] is None else p["Gw2"]
        self.improved, self.g = p["scheme"] == "improved", p["g"]
        self.stencil = [e for e in itertools.product(range(-2, 3), repeat=d) if _sq(e) in self.G]
        # adhesion vector, and the second layer's first-layer partners: {partner: coefficient per axis} at wall nodes
        a = [torch.zeros(solid.shape, dtype=torch.float64, device=dev) for _ in range(d)]
        near = torch.zeros_like(solid)
        for e in self.stencil:
            near |= self.at(self.nofluid, e)
        self.wall = (near & self.fluid).nonzero(as_tuple=True)
        coef = {}
        for e in self.stencil:
            w = self.G[_sq(e)]
            if max(abs(v) for v in e) < 2:
                s = self.at(self.solid1, e)
            else:
                nf, pe = self.at(self.nofluid, e), _sgn(e)
                s = nf & self.at(self.solid1, e if p["second_layer"] == "psi" else pe)
                c = coef.setdefault(pe, [0.0] * d)
                for k in range(d):
                    if e[k]:
                        c[k] = c[k] + w * e[k] * nf[self.wall].double()
            if p["adhesion_stencil"] == "e8":
                for k in range(d):
                    if e[k]:
                        a[k] += w * e[k] * s.double()
        if p["adhesion_stencil"] != "e8":
            for e in self.E[1:]:
                for k in range(d):
                    if e[k]:
                        a[k] += self.W[_sq(e)] * e[k] * self.at(self.solid1, e).double()
        self.a, self.coef = a, coef
        # blocked links: the node upstream along e_i is not fluid (outside an open column: the boundary rule)
        block = self.pad(solid, True, clamp=True)
        self.blocked = [self.at(block, tuple(-v for v in e)) for e in self.E]

    def axis(self, k):
        return self.d - 1 - k  # x is the last array axis

    def pad(self, t, outside, clamp):
        for k in range(self.d):
            ax, n = self.axis(k), t.shape[self.axis(k)]
            if self.bc[k] == "periodic":
                lo, hi = t.narrow(ax, n - 2, 2), t.narrow(ax, 0, 2)
            elif self.bc[k] == "open" and clamp:
                lo = torch.cat([t.narrow(ax, 0, 1)] * 2, ax)
                hi = torch.cat([t.narrow(ax, n - 1, 1)] * 2, ax)
            else:
                lo = hi = torch.full_like(t.narrow(ax, 0, 2), outside)
            t = torch.cat([lo, t, hi], ax)
        return t

    def at(self, padded, e):
        """The padded array's values at x + e, for every x of the lattice."""
        for k in range(self.d):
            ax = self.axis(k)
            padded = padded.narrow(ax, 2 + e[k], self.solid.shape[ax])
        return padded

    def feq0(self, rho):
        return torch.stack([self.W[_sq(e)] * rho for e in self.E])

    def inlet_rows(self):
        ny, u = self.sc.ny, self.sc.u_in
        y = torch.arange(ny, dtype=torch.float64, device=self.dev) + 0.5
        return u * 4 * y * (ny - y) / ny ** 2 if self.sc.inlet_profile == "poiseuille" else torch.full_like(y, u)

    def open_x(self, fs, f):
        """Inlet at x = 0 (non-equilibrium bounce-back) and copy outflow at x = nx - 1 (f: [2][9][ny][nx])."""
        if self.bc[0] != "open":
            return f
        u, fl0, fl1 = self.inlet_rows(), self.fluid[:, 0], self.fluid[:, -1]
        up = self.fluid[:, -2]
        new = f.clone()
        for k in range(2):
            for i, e in enumerate(self.E):
                if e[0] > 0:
                    v = f[k, self.opp[i], :, 0] + 6 * self.W[_sq(e)] * self.sc.rho_in[k] * u
                    new[k, i, :, 0] = torch.where(fl0, v, f[k, i, :, 0])
                elif e[0] < 0:
                    v = torch.where(up, f[k, i, :, -2], fs[k, self.opp[i], :, -1])
                    new[k, i, :, -1] = torch.where(fl1, v, f[k, i, :, -1])
        return new

    def start(self, rA, rB):
        f = torch.stack([self.feq0(torch.where(self.fluid, r, torch.zeros_like(r))) for r in (rA, rB)])
        return self.open_x(f, f)

    def macro(self, f):
        """Densities, forces [2][d] and velocity [d] (0 velocity at solid nodes)."""
        rho = f.sum(1)
        grads = []
        for k in range(2):
            pr = self.pad(rho[k], 0.0, clamp=True)
            free = pr * ~self.nofluid
            g = [torch.zeros_like(rho[k]) for _ in range(self.d)]
            for e in self.stencil:
                v = self.at(free if max(abs(x) for x in e) == 2 else pr, e)
                for j in range(self.d):
                    if e[j]:
                        g[j].add_(v, alpha=self.G[_sq(e)] * e[j])
            for pe, c in self.coef.items():
                v = self.at(pr, pe)[self.wall]
                for j in range(self.d):
                    if torch.is_tensor(c[j]):
                        g[j].index_put_(self.wall, c[j] * v, accumulate=True)
            grads.append(g)
        rA, rB = rho[0], rho[1]
        tot = torch.where(self.fluid, rA + rB, torch.ones_like(rA))
        if self.improved:
            re, l, dl = (rA - rB) / tot, self.lam, self.delta
            s1 = 2 * l / (1 + l)
            hi = s1 + 2 * (l * l - l) / (dl * (1 + l)) * re + (l - l * l) / (dl * dl * (1 + l)) * re * re
            lo = s1 + 2 * (l - 1) / (dl * (1 + l)) * re + (l - 1) / (dl * dl * (1 + l)) * re * re
            one = torch.ones_like(re)
            GA = self.Gw2 * torch.where(re > dl, l * one, torch.where(re > 0, hi, torch.where(re > -dl, lo, one)))
        else:
            GA = self.lam * self.Gw2
        F = [[], []]
        u = []
        for j in range(self.d):
            FA = -self.Gc * rA * grads[1][j] - GA * rA * self.a[j] + rA * self.g[j]
            FB = -self.Gc * rB * grads[0][j] - self.Gw2 * rB * self.a[j] + rB * self.g[j]
            mom = sum(e[j] * (f[0, i] + f[1, i]) for i, e in enumerate(self.E) if e[j])
            F[0].append(FA)
            F[1].append(FB)
            u.append(torch.where(self.fluid, (mom + 0.5 * (FA + FB)) / tot, torch.zeros_like(rA)))
        return rho, F, u

    def step(self, f):
        rho, F, u = self.macro(f)
        usq = sum(v * v for v in u)
        fs = torch.empty_like(f)
        for k in range(2):
            uF = sum(a * b for a, b in zip(u, F[k]))
            cF = 1 - 0.5 / self.tau[k]
            for i, e in enumerate(self.E):
                w = self.W[_sq(e)]
                eu = sum(e[j] * u[j] for j in range(self.d) if e[j]) if i else torch.zeros_like(usq)
                eF = sum(e[j] * F[k][j] for j in range(self.d) if e[j]) if i else torch.zeros_like(usq)
                fe = w * rho[k] * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * usq)
                fs[k, i] = f[k, i] + (fe - f[k, i]) / self.tau[k] + cF * w * (3 * (eF - uF) + 9 * eu * eF)
        fs *= self.fluid
        new = torch.empty_like(f)
        walls = getattr(self.sc, "u_wall", (0.0, 0.0))
        for i, e in enumerate(self.E):
            moved = fs[:, i]
            for j in range(self.d):
                if e[j]:
                    moved = torch.roll(moved, e[j], 1 + self.axis(j))
            new[:, i] = torch.where(self.blocked[i], fs[:, self.opp[i]], moved)
            if self.d == 2 and self.bc[1] == "wall" and e[1] and e[0]:
                row, uw = (0, walls[0]) if e[1] > 0 else (-1, walls[1])
                if uw:
                    new[:, i, row] += 6 * self.W[_sq(e)] * e[0] * uw * fs[:, :, row].sum(1)
        new *= self.fluid
        return self.open_x(fs, new)

    def diag(self, rho, u):
        fl = self.fluid
        tot = rho[0] + rho[1]
        speed = torch.sqrt(sum(v * v for v in u))[fl].max()
        ext = [getattr(rho[k][fl], op)() for k in range(2) for op in ("min", "max")]
        return [float(v) for v in [rho[0].sum(), rho[1].sum(), *[(tot * v).sum() for v in u], speed, *ext]], int(fl.sum())

    def angle(self, rho, surface):
        """Contact angle and rms residual: zeros of rho^e along lattice lines, Kasa fit, one Gauss-Newton step."""
        near = self.solid
        for k in range(self.d):  # no non-fluid site within three cells
            ax = self.axis(k)
            pads = []
            for s in range(-3, 4):
                m = torch.roll(near, s, ax)
                if self.bc[k] != "periodic" and s:
                    m.narrow(ax, 0 if s > 0 else near.shape[ax] + s, abs(s)).fill_(True)
                pads.append(m)
            near = torch.stack(pads).any(0)
        use = ~near
        phi = (rho[0] - rho[1]) / torch.where(self.fluid, rho[0] + rho[1], torch.ones_like(rho[0]))
        pts = []
        for k in range(self.d):
            ax, n = self.axis(k), phi.shape[self.axis(k)]
            a, b = phi.narrow(ax, 0, n - 1), phi.narrow(ax, 1, n - 1)
            hit = use.narrow(ax, 0, n - 1) & use.narrow(ax, 1, n - 1) & ((a > 0) != (b > 0))
            at = hit.nonzero().double().flip(1)
            at[:, k] += a[hit] / (a[hit] - b[hit])
            pts.append(at)
        p = torch.cat(pts)
        m = p.mean(0)
        q = p - m
        A = torch.cat([2 * q, torch.ones_like(q[:, :1])], 1)
        x = torch.linalg.solve(A.T @ A, A.T @ (q * q).sum(1))
        c, r = m + x[:-1], torch.sqrt(x[-1] + (x[:-1] ** 2).sum())
        dist = (p - c).norm(dim=1)
        J = torch.cat([-(p - c) / dist[:, None], -torch.ones_like(dist[:, None])], 1)
        x = torch.linalg.solve(J.T @ J, -J.T @ (dist - r))
        c, r = c + x[:-1], float(r + x[-1])
        rms = float((((p - c).norm(dim=1) - r) ** 2).mean().sqrt())
        if "y_w" in surface:
            cth = -surface.get("normal", 1) * (float(c[1]) - surface["y_w"]) / r
        else:
            o = surface.get("c") or (surface["cx"], surface["cy"])
            d2 = sum((float(c[k]) - o[k]) ** 2 for k in range(self.d))
            cth = (surface["R"] ** 2 + r * r - d2) / (2 * r * surface["R"])
        return math.degrees(math.acos(max(-1.0, min(1.0, cth)))), rms


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    fields, diags, counts, angles = [], [], [], []
    for sc in _scenarios(case, seed):
        ex = _Exact(sc, dev)
        f = ex.start(*[torch.from_numpy(r).to(dev) for r in (sc.rhoA0, sc.rhoB0)])
        for _ in range(case["steps"]):
            f = ex.step(f)
        rho, _, u = ex.macro(f)
        fields.append(torch.stack([rho[0], rho[1], *u]).reshape(2 + ex.d, -1))
        if case["read"] in ("all", "diagnostics"):
            d, n = ex.diag(rho, u)
            diags.append(d)
            counts.append(n)
        if case["read"] == "all":
            angles.append(ex.angle(rho, sc.sphere if case["kind"] == "sphere" else sc.surface))
    res = {"fields": torch.cat(fields, 1)}
    if diags:
        one = case["kind"] == "sphere"
        res["diag"], res["n_fluid"] = torch.tensor(diags[0] if one else diags, dtype=torch.float64), counts[0] if one else torch.tensor(counts)
    if angles:
        a = torch.tensor(angles, dtype=torch.float64)
        res["angle"] = a[0] if case["kind"] == "sphere" else a.T.contiguous()
    return res
