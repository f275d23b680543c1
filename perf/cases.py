"""The workloads whose speed is watched, each through the library's C ABI.

A case is one rotating vessel (or an uneven ensemble of them), one form of the
step (FP64 or mixed) and what a program does with it in one pass:

* ``advance``: some time steps, then the state read out to device arrays (one
  output frame of a run);
* ``monitor``: the same with the conservation totals read back after every
  step (a run that watches its budgets);
* ``evaluate``: a context made anew on the kept buffers from device arrays of
  positions, velocities and spins (neighbour lists, density, pressure, pair
  forces of a given configuration: the start of a job), then the fields read
  out.

The vessels are jittered lattices in rigid rotation with a random species draw
and a little velocity noise, with two dummy layers behind the inner wall
wherever a pass is repeated for long.  The mixed form stores and computes its
fields in FP32; its results are handed on as FP32 here (the library's read-out
widens them to double), those of the FP64 form as FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2405_03980_gb300 import _binding as B

DEVICE = "cuda:0"
FIELDS = ("pos", "vel", "spin", "rho", "P", "acc", "dspin")
WIDTH = {"pos": 3, "vel": 3, "spin": 3, "rho": 1, "P": 1, "acc": 3, "dspin": 3}
FLAGS = {"": B.SPH_FLAGS_DEFAULT,
         "filter": B.SPH_FLAGS_DEFAULT | B.SPH_PFILTER,
         "collision": B.SPH_FLAGS_DEFAULT | B.SPH_COLLISION,
         "filter+collision": B.SPH_FLAGS_DEFAULT | B.SPH_PFILTER | B.SPH_COLLISION}


def _vessel(name, form, do, steps, R, H, Omega=0.1, f_v=0.3, dummy=2, extras=""):
    return {"name": name, "form": form, "do": do, "steps": steps, "R": R, "H": H,
            "Omega": Omega, "f_v": f_v, "dummy": dummy, "extras": extras}


def listed():
    return [
        # parity-size runs and parameter studies: launches and latency count
        _vessel("small vessel, mixed", "mixed", "advance", 10, 10.0, 20),
        _vessel("small vessel, fp64", "fp64", "advance", 5, 10.0, 20),
        # a ragged mid-size vessel: odd radius and height, cells that do not
        # divide the box evenly
        _vessel("ragged vessel, mixed", "mixed", "advance", 8, 23.7, 41, Omega=0.17, f_v=0.12),
        # a run that checks its angular-momentum and mass budgets every step
        _vessel("monitored vessel, fp64", "fp64", "monitor", 2, 28.0, 56),
        # the paper's 2.4M resolution, both forms
        _vessel("2.4M vessel, mixed", "mixed", "advance", 8, 72.5, 145),
        _vessel("2.4M vessel, fp64", "fp64", "advance", 2, 72.5, 145),
        # the start of a job from given arrays: the list build counts in full;
        # the low-temperature (near-inviscid) vessel
        _vessel("low-T job start, mixed", "mixed", "evaluate", 0, 72.5, 145, Omega=0.2, f_v=0.01),
        _vessel("ragged job start, fp64", "fp64", "evaluate", 0, 41.3, 63, Omega=0.07, f_v=0.45),
        # Algorithm 1 with both optional steps on the paper's own vessel shape
        _vessel("8.6M paper vessel, mixed", "mixed", "advance", 5, 190.0, 76, f_v=1.0 / 6.0,
                extras="filter+collision"),
        # parameter sweep: 64 uneven independent vessels in one launch per stage
        {"name": "ensemble of 64, mixed", "form": "mixed", "do": "advance", "steps": 5,
         "members": 64, "sizes": 1234, "n_lo": 2e4, "n_hi": 5e5, "extras": ""},
        # the paper's 19.6M resolution, both forms: the headline workload
        _vessel("19.6M vessel, mixed", "mixed", "advance", 8, 146.0, 292, dummy=1),
        _vessel("19.6M vessel, fp64", "fp64", "advance", 2, 146.0, 292, dummy=1),
    ]


def draw(rng):
    """A vessel of 6e3 to 1.9e7 fluid particles, its shape, speed, species mix,
    form and options drawn over what the listed ones span."""
    form = rng.choice(["mixed", "mixed", "fp64"])
    n_max = 1.9e7 if form == "mixed" else 4e6
    nf = math.exp(rng.uniform(math.log(6e3), math.log(n_max)))
    rh = math.exp(rng.uniform(math.log(0.25), math.log(2.5)))
    H = max(11, int(round((nf / (math.pi * rh * rh)) ** (1.0 / 3.0))))
    R = max(6.0, round(math.sqrt(nf / (math.pi * H)), 1))
    do = rng.choice(["advance", "advance", "advance", "evaluate"])
    if form == "fp64" and rng.random() < 0.25:
        do = "monitor"
    steps = rng.randint(2, 8) if form == "mixed" else rng.randint(1, 4)
    steps = {"evaluate": 0, "monitor": min(steps, 2)}.get(do, steps)
    extras = rng.choice(["", "", "", "filter", "collision", "filter+collision"])
    return {"form": form, "do": do, "steps": steps, "R": R, "H": H,
            "Omega": round(rng.uniform(0.05, 0.2), 3), "f_v": round(rng.uniform(0.01, 0.5), 3),
            "dummy": 2, "extras": extras}


# ------------------------------------------------------------------- vessels

def _members(case):
    """(R, H, Omega, f_v, dummy layers) of every vessel of the case."""
    if "members" not in case:
        return [(case["R"], case["H"], case["Omega"], case["f_v"], case["dummy"])]
    rng = np.random.Generator(np.random.PCG64(case["sizes"]))
    out = []
    for _ in range(case["members"]):
        nf = math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))
        om, fv, rh = rng.uniform(0.05, 0.2), rng.uniform(0.02, 0.5), rng.uniform(0.25, 1.0)
        R = (nf * rh / math.pi) ** (1.0 / 3.0)
        out.append((R, max(8, int(round(R / rh))), om, fv, 2))
    return out


def _disc(R, dummy):
    """Lattice points of one layer, x-major, and their kind: 0 fluid, 2 inner
    wall, 3 dummy."""
    m = int(math.ceil(R + 1 + dummy)) + 1
    ax = np.arange(-m, m, dtype=np.float64) + 0.5
    X, Y = (a.ravel() for a in np.meshgrid(ax, ax, indexing="ij"))
    r = np.sqrt(X * X + Y * Y)
    kind = np.full(X.shape, -1, dtype=np.int64)
    kind[r < R] = 0
    kind[(r >= R) & (r < R + 1)] = 2
    kind[(r >= R + 1) & (r < R + 1 + dummy)] = 3
    keep = kind >= 0
    return X[keep], Y[keep], kind[keep]


def _params(R, H, Omega, dummy):
    """Dimensionless recipe of the workloads: c_s = 10 Omega R, Re = 100,
    dt = h / (4 c_s), h = 1.3, lattice spacing and rest density 1."""
    h = 1.3
    cs = 10.0 * Omega * R
    p0 = cs * cs / 7.0
    eta = Omega * R * R / 100.0
    ext = R + (1 + dummy) + 2.0 * h
    return dict(dx=1.0, h=h, rho0=1.0, alpha_P=7.0, p0=p0, beta_P=p0, eta_bar=eta, eta_r=eta,
                xi_bar=0.0, C_l=1e-3 * Omega, C_T=0.01 * p0, C_omega=0.016, mass_ratio=1.0,
                inertia_coef=0.1, Omega=Omega, dt=0.25 * h / cs, col_dist=0.8, col_e=0.2,
                box_lo=(-ext, -ext, 0.0), box_hi=(ext, ext, float(H)), periodic_z=1)


def _vessel_arrays(R, H, Omega, f_v, dummy, gen):
    """Positions, velocities, spins and species of one vessel on the GPU."""
    X, Y, kind = (torch.as_tensor(a, device=DEVICE) for a in _disc(R, dummy))
    nl = X.numel()
    n = nl * H
    pos = torch.empty((n, 3), dtype=torch.float64, device=DEVICE)
    pos[:, 0] = X.repeat(H)
    pos[:, 1] = Y.repeat(H)
    pos[:, 2] = (torch.arange(H, dtype=torch.float64, device=DEVICE) + 0.5).repeat_interleave(nl)
    sp = kind.to(torch.uint8).repeat(H)
    fluid = (sp == 0)[:, None].to(torch.float64)
    viscous = torch.rand(n, generator=gen, device=DEVICE, dtype=torch.float64) < f_v
    jitter = torch.rand((n, 3), generator=gen, device=DEVICE, dtype=torch.float64)
    noise = torch.randn((n, 3), generator=gen, device=DEVICE, dtype=torch.float64)
    pos += fluid * (jitter - 0.5) * 0.1
    vel = torch.stack([-Omega * pos[:, 1], Omega * pos[:, 0], torch.zeros_like(pos[:, 0])], 1)
    vel += fluid * noise * 1e-3
    spin = torch.zeros_like(pos)
    spin[:, 2] = Omega * (1.0 - fluid[:, 0])
    sp[(sp == 0) & viscous] = 1
    return pos, vel, spin, sp


def _arrays(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    parts = [_vessel_arrays(*m, gen) for m in _members(case)]
    counts = [int(p[3].numel()) for p in parts]
    if len(parts) == 1:
        return counts, parts[0]
    return counts, tuple(torch.cat([p[k] for p in parts]).contiguous() for k in range(4))


# ---------------------------------------------------------------------- runs

class _Run:
    """The buffers and the context that a program keeps."""

    def __init__(self, case, seed):
        self.do, self.steps, self.form = case["do"], case["steps"], case["form"]
        self.params = []
        for R, H, om, _, dummy in _members(case):
            p = _params(R, H, om, dummy)
            p["flags"] = FLAGS[case["extras"]]
            p["precision"] = B.SPH_MIXED if self.form == "mixed" else B.SPH_FP64
            self.params.append(B.params_from_dict(p))
        self.counts, arrays = _arrays(case, seed)
        n = sum(self.counts)
        self.ctx = None
        self.state = torch.empty(B.sph_state_bytes(self.params, self.counts), dtype=torch.uint8,
                                 device=DEVICE)
        self.work = torch.empty(B.sph_workspace_bytes(self.params, self.counts),
                                dtype=torch.uint8, device=DEVICE)
        names = FIELDS[3:] if self.do == "evaluate" else FIELDS
        self.out = {k: torch.empty((n, 3) if WIDTH[k] == 3 else n, dtype=torch.float64,
                                   device=DEVICE) for k in names}
        if self.do == "evaluate":
            self.arrays = arrays
        else:
            self.open(arrays)

    def open(self, arrays):
        self.close()
        self.ctx = B.sph_init_batch(self.params, self.counts, *arrays, self.state,
                                    self.state.numel(), self.work, self.work.numel(),
                                    torch.cuda.current_stream().cuda_stream)

    def read(self):
        B.sph_get_state(self.ctx, **self.out)
        if self.form == "mixed":
            return {k: v.to(torch.float32) for k, v in self.out.items()}
        return dict(self.out)

    def close(self):
        if self.ctx is not None:
            B.sph_destroy(self.ctx)
            self.ctx = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def prepare(case, seed):
    return _Run(case, seed)


def run(state):
    if state.do == "evaluate":
        state.open(state.arrays)
        return state.read()
    if state.do == "monitor":
        totals = []
        for _ in range(state.steps):
            B.sph_step(state.ctx, 1)
            totals.append(B.sph_diagnostics(state.ctx))
        return {"totals": totals, **state.read()}
    B.sph_step(state.ctx, state.steps)
    return state.read()


def work(case):
    """One pass: per step every particle's position, velocity, spin and species
    read and written once, the accelerations, densities and pressures written;
    per unique pair within the kernel support (39 per particle on the lattice)
    the operations of the density sum and of the terms the pair's species
    carry; an evaluation reads the arrays and writes the fields."""
    b = f = 0.0
    word = 4.0 if case["form"] == "mixed" else 8.0
    passes = max(case["steps"], 1)
    for R, H, _, fv, dummy in _members(case):
        n = float(_disc(R, dummy)[0].size * H)
        pair = 18.0 + (1 - fv) ** 2 * 23.0 + 2 * fv * (1 - fv) * 76.0 + fv * fv * 79.0
        if "filter" in case["extras"]:
            pair += 8.0
        if case["do"] == "evaluate":
            b += n * (9 * 8.0 + 1.0 + 8 * word)
        else:
            b += n * (passes * (2 * (9 * word + 1.0) + 8 * word) + 17 * word)
        f += n * passes * 39.0 * pair
    return {"bytes": b, "flops": f}


# --------------------------------------------- the same in 64 bits with torch

def _kernel_constants(p):
    h = p["h"]
    aD = 21.0 / (16.0 * math.pi * h ** 3)
    total = 0.0
    for a in range(-3, 4):
        for b in range(-3, 4):
            for c in range(-3, 4):
                q = math.sqrt(a * a + b * b + c * c) / h
                if q < 2.0:
                    total += aD * (1 - 0.5 * q) ** 4 * (2 * q + 1)
    return aD, p["rho0"] / total  # equal particle masses (mass_ratio 1)


class _Exact:
    """One vessel stepped in torch float64 over explicit pair lists."""

    ROWS = 400_000

    def __init__(self, p, extras, pos, vel, spin, sp):
        self.p, self.extras = p, extras
        self.pos, self.vel, self.spin, self.sp = pos.clone(), vel.clone(), spin.clone(), sp
        self.aD, self.m = _kernel_constants(p)
        self.theta = 0.0
        self.ref = pos[:, :2].clone()
        self.wall = (sp >= 2)[:, None]
        self.T = torch.zeros(3, dtype=torch.float64, device=pos.device)
        self.J = torch.zeros_like(self.T)
        self.place()
        self.evaluate()

    def place(self):
        c, s, om = math.cos(self.theta), math.sin(self.theta), self.p["Omega"]
        x, y = c * self.ref[:, 0] - s * self.ref[:, 1], s * self.ref[:, 0] + c * self.ref[:, 1]
        z = self.pos[:, 2]
        o = torch.zeros_like(x)
        self.pos = torch.where(self.wall, torch.stack([x, y, z], 1), self.pos)
        self.vel = torch.where(self.wall, torch.stack([-om * y, om * x, o], 1), self.vel)
        self.spin = torch.where(self.wall, torch.stack([o, o, o + om], 1), self.spin)

    def pairs(self):
        """Blocks of (i, j, r_ij) over all neighbours j != i of the rows that
        sum a density."""
        p = self.p
        cut, Hz = 2.0 * p["h"], p["box_hi"][2] - p["box_lo"][2]
        lo, ext = p["box_lo"][0], p["box_hi"][0] - p["box_lo"][0]
        nx = int(ext / cut) + 2
        nz = int(Hz / cut)
        if nz < 3:
            raise ValueError("vessel too flat")
        cx, cy = (((self.pos[:, a] - lo) / (ext / (nx - 2))).floor().long().clamp(0, nx - 3) + 1
                  for a in (0, 1))
        cz = (self.pos[:, 2] / (Hz / nz)).floor().long().clamp(0, nz - 1)
        key = (cz * nx + cy) * nx + cx
        order = torch.argsort(key, stable=True)
        ks = key[order]
        start = torch.searchsorted(ks, torch.arange(nx * nx * nz + 2, device=ks.device))
        ps = self.pos[order]
        rows = torch.nonzero(self.sp[order] != 3)[:, 0]
        for r0 in range(0, rows.numel(), self.ROWS):
            row = rows[r0:r0 + self.ROWS]
            got = []
            for dz in (-1, 0, 1):
                z2 = cz[order[row]] + dz
                shift = torch.where(z2 < 0, -Hz, torch.where(z2 >= nz, Hz, 0.0)).to(ps.dtype)
                z2 = z2 % nz
                for dy in (-1, 0, 1):
                    k0 = (z2 * nx + cy[order[row]] + dy) * nx + cx[order[row]] - 1
                    s0, s1 = start[k0], start[k0 + 3]
                    t = torch.arange(int((s1 - s0).max()), device=ks.device)
                    j = s0[:, None] + t
                    ok = j < s1[:, None]
                    j = torch.where(ok, j, s0[:, None].clamp(max=ks.numel() - 1))
                    i = row[:, None].expand_as(j)
                    a, b, ok = i[ok], j[ok], None
                    d = ps[a] - ps[b]
                    d[:, 2] -= shift[:, None].expand(-1, t.numel())[(s0[:, None] + t) < s1[:, None]]
                    near = (d.square().sum(1) < cut * cut) & (a != b)
                    got.append((order[a[near]], order[b[near]], d[near]))
            yield tuple(torch.cat([g[k] for g in got]) for k in range(3))

    def evaluate(self):
        p, n, m = self.p, self.sp.numel(), self.m
        h, aD = p["h"], self.aD
        zero = torch.zeros(n, dtype=torch.float64, device=self.pos.device)
        shape = lambda q: (1 - 0.5 * q) ** 4 * (2 * q + 1)  # noqa: E731
        lists = list(self.pairs())
        rho = zero + m * aD
        for i, j, d in lists:
            rho.index_add_(0, i, m * aD * shape(d.square().sum(1).sqrt() / h))
        rho = torch.where(self.sp == 3, torch.full_like(rho, p["rho0"]), rho)
        P = p["p0"] * (rho / p["rho0"]) ** 7 - p["beta_P"]
        V = m / rho
        if "filter" in self.extras:
            num, den = V * P, V.clone()
            for i, j, d in lists:
                w = torch.where(self.sp[j] == 3, 0.0, V[j] * shape(d.square().sum(1).sqrt() / h))
                num.index_add_(0, i, w * P[j])
                den.index_add_(0, i, w)
            P = torch.where(self.sp == 3, P, num / den)
        self.rho, self.P = rho, P
        Pr = P / rho ** 2
        F_acc = torch.zeros((n, 3), dtype=torch.float64, device=self.pos.device)
        tau = torch.zeros_like(F_acc)
        T = torch.zeros(3, dtype=torch.float64, device=self.pos.device)
        A, Bv = 10.0 * (p["eta_bar"] - 0.6 * p["eta_r"]), 4.0 * p["eta_r"]
        for i, j, d in lists:
            keep = self.sp[i] < 2
            i, j, d = i[keep], j[keep], d[keep]
            r2 = d.square().sum(1)
            q = r2.sqrt() / h
            F = 5.0 * aD / (h * h) * (1 - 0.5 * q) ** 3
            W = aD * shape(q)
            unlike = ((self.sp[i] == 0) != (self.sp[j] == 0)).to(d.dtype)
            both = ((self.sp[i] != 0) & (self.sp[j] != 0)).to(d.dtype)
            VV = V[i] * V[j]
            v = self.vel[i] - self.vel[j]
            u = v + 0.5 * torch.linalg.cross(d, self.spin[i] + self.spin[j])
            dv = (d * v).sum(1)
            central = m * m * (Pr[i] + Pr[j]) * F + (Bv - A) * both * VV * F * dv / r2
            if "collision" in self.extras:
                hit = (r2 < p["col_dist"] ** 2) & (dv < 0)
                central -= torch.where(hit, (1 + p["col_e"]) * 0.5 * m * dv / r2 / p["dt"], 0.0)
            turn = (-Bv * both * VV * F - p["C_l"] * unlike * VV * W)[:, None] * u
            f = central[:, None] * d + turn
            f[:, :2] += (p["C_T"] * unlike * VV * F)[:, None] * d[:, :2]
            t = -0.5 * torch.linalg.cross(d, turn)
            F_acc.index_add_(0, i, f)
            tau.index_add_(0, i, t)
            w = self.sp[j] >= 2
            T += (torch.linalg.cross(self.pos[i[w]], f[w]) + t[w]).sum(0)
        self.acc, self.dspin = F_acc / m, tau / (p["inertia_coef"] * m * p["dx"] ** 2)
        self.T_old, self.T = self.T, T

    def step(self):
        p = self.p
        half = 0.5 * p["dt"]
        fluid = ~self.wall
        self.vel = torch.where(fluid, self.vel + half * self.acc, self.vel)
        self.spin = torch.where(fluid, self.spin + half * self.dspin, self.spin)
        self.pos = torch.where(fluid, self.pos + p["dt"] * self.vel, self.pos)
        Hz = p["box_hi"][2] - p["box_lo"][2]
        z = self.pos[:, 2]
        self.pos[:, 2] = torch.where(z >= Hz, z - Hz, torch.where(z < 0, z + Hz, z))
        self.theta += p["Omega"] * p["dt"]
        self.place()
        self.evaluate()
        self.vel = torch.where(fluid, self.vel + half * self.acc, self.vel)
        self.spin = torch.where(fluid, self.spin + half * self.dspin, self.spin)
        self.J += half * (self.T_old + self.T)

    def totals(self, n_pairs=None):
        p, fl, m = self.p, self.sp < 2, self.m
        pos, v, w, rho = (a[fl] for a in (self.pos, self.vel, self.spin, self.rho))
        inertia = p["inertia_coef"] * m * p["dx"] ** 2
        energy = (p["p0"] / 6.0 * ((rho / p["rho0"]) ** 6 - 1.0)
                  + p["beta_P"] * (1.0 / rho - 1.0 / p["rho0"]))
        n_s, n_n = int((self.sp == 0).sum()), int((self.sp == 1).sum())
        return {"mass": m * (n_s + n_n), "mass_s": m * n_s, "mass_n": m * n_n,
                "mom": (m * v).sum(0).tolist(),
                "L_orb": (m * torch.linalg.cross(pos, v)).sum(0).tolist(),
                "L_spin": (inertia * w).sum(0).tolist(),
                "E_kin": 0.5 * m * float(v.square().sum()),
                "E_rot": 0.5 * inertia * float(w.square().sum()),
                "E_int": m * float(energy.sum()),
                "T_wall": self.T.tolist(), "J_wall": self.J.tolist(),
                "rho_min": float(rho.min()), "rho_max": float(rho.max()),
                "v_max": float(v.square().sum(1).max().sqrt()),
                "n_pairs": None, "step": None, "theta": self.theta}


def exact(case, seed):
    counts, arrays = _arrays(case, seed)
    if sum(counts) * (case["steps"] + 1) > 3.0e7 or len(counts) > 8:
        return None
    sims, at, totals = [], 0, []
    for n, (R, H, om, _, dummy) in zip(counts, _members(case)):
        sims.append(_Exact(_params(R, H, om, dummy), case["extras"],
                           *(a[at:at + n] for a in arrays)))
        at += n
    for s in sims:
        for _ in range(case["steps"]):
            s.step()
            if case["do"] == "monitor":
                totals.append(s.totals())
    names = FIELDS[3:] if case["do"] == "evaluate" else FIELDS
    out = {k: torch.cat([getattr(s, k) for s in sims]) for k in names}
    fluid = arrays[3] < 2
    for k in ("acc", "dspin"):
        out[k] = out[k] * fluid[:, None]
    return {"totals": totals, **out} if case["do"] == "monitor" else out
