"""Performance cases: what a program does with this engine, call by call.

Every case is one engine (``capi.Engine``) that a program has created, filled
with spheres and keeps; one pass is the call sequence of its time loop:

* ``drag``     a few fixed spheres in a small periodic box with a body force
               (drag measurement): steps, then the forces and torques;
* ``settle``   spheres settling in a periodic box under gravity with the device
               DEM: steps, then forces, torques and the particle state (and,
               where asked, the density and velocity field, as a field dump);
* ``channel``  a bed of fixed spheres between walls with a body force: the
               spheres are mapped once, then steps and forces;
* ``bed``      the fluidized bed: no-slip side walls, velocity inflow at the
               bottom, pressure outflow at the top, SRT, the linear
               approximation, free spheres;
* ``coupled``  the settling box driven by a program that owns the particles:
               their state goes in before each step, forces and the new state
               come out after it;
* ``train``    the surrogate's training on the device.

Spheres sit in the cells of a regular lattice with a random offset (gap at
least ``gap``), drawn from the seed, as do their velocities; the fluid starts
at rest (``drag``: with noise).  ``exact`` is the same time loop in plain FP64
torch, dense over the grid.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2303_11811_gb300 import capi

CX = (0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0)
CY = (0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1)
CZ = (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1)
W = (1.0 / 3.0,) + (1.0 / 18.0,) * 6 + (1.0 / 36.0,) * 12
MAGIC = 3.0 / 16.0
REACH = math.sqrt(3.0) / 2.0


def _case(name, kind, nx, ny, nz, steps, precision="fp64", streaming="pull",
          eps="supersample", eps_n=8, phi=0.15, rmin=3.0, rmax=6.0, field=False):
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, steps=steps, precision=precision,
                streaming=streaming, eps=eps, eps_n=eps_n, phi=phi, rmin=rmin, rmax=rmax,
                field=field)


def listed():
    return [
        # the smallest call: one step of the 32^3 box with one sphere, then its force
        _case("drag32_1step", "drag", 32, 32, 32, 1, eps_n=4, phi=0.008, rmin=4.0, rmax=4.0),
        # the 128^3 settling box (400 spheres r = 6, 4^3 sampling), with a field dump
        _case("settle128_fields", "settle", 128, 128, 128, 50, eps_n=4, phi=0.173, rmin=6.0,
              field=True),
        # a program that owns the particles, 256^3, one step per exchange
        _case("coupled256", "coupled", 256, 256, 256, 1),
        # the plain FP64 method on a large settling box (half of the 512x512x1024 one)
        _case("settle512_fp64", "settle", 512, 512, 512, 5),
        # the fast form of the full settling box: FP32 deviations in place, surrogate
        _case("settle512_fp32_mlp", "settle", 512, 512, 1024, 10, precision="fp32",
              streaming="aa", eps="mlp"),
        # the double-float form
        _case("settle256_df64", "settle", 256, 256, 256, 10, precision="df64"),
        # a ragged FP64 channel of fixed spheres
        _case("channel_fp64_ragged", "channel", 203, 131, 301, 20, phi=0.20, rmin=5.0, rmax=5.0),
        # the channel workload in FP32
        _case("channel_fp32", "channel", 256, 256, 512, 20, precision="fp32", phi=0.20, rmin=5.0,
              rmax=5.0),
        # the same method in place on a ragged grid
        _case("channel_fp32_aa_ragged", "channel", 250, 190, 310, 20, precision="fp32",
              streaming="aa", eps_n=4, phi=0.20, rmin=5.0, rmax=5.0),
        # the fluidized bed, dilute in FP64 and dense in FP32
        _case("bed_dilute_fp64", "bed", 500, 200, 800, 5, eps="linear", phi=0.033, rmin=10.0,
              rmax=10.0),
        _case("bed_dense_fp32", "bed", 500, 200, 800, 10, precision="fp32", eps="linear", phi=0.40,
              rmin=10.0, rmax=10.0),
        # training of the surrogate: 2^18 samples, one epoch
        dict(name="train_2e18", kind="train", samples=1 << 18, epochs=1, batch=1024),
    ]


def draw(rng):
    def loguni(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["drag", "settle", "settle", "settle", "channel", "channel", "bed", "bed",
                       "coupled", "train"])
    if kind == "train":
        return dict(kind=kind, samples=loguni(1 << 14, 1 << 18), epochs=rng.randint(1, 3),
                    batch=rng.choice([512, 1024, 2048]))
    precision = rng.choice(["fp64", "fp64", "fp32", "fp32", "df64"])
    streaming = "pull" if kind == "bed" else rng.choice(["pull", "pull", "aa"])
    eps, eps_n = rng.choice([("supersample", 4), ("supersample", 8), ("supersample", 8),
                             ("linear", 8), ("mlp", 8)])
    if kind == "drag":
        n = [rng.randint(24, 96) for _ in range(3)]
        steps, r, phi = rng.choice([1, 1, 10, 50]), rng.uniform(3.0, 5.0), rng.uniform(0.005, 0.1)
        rmin = rmax = r
    else:
        n = [loguni(48, 512) for _ in range(3)]
        cells = n[0] * n[1] * n[2]
        # a pass costs no more than the largest listed ones
        steps = max(1, min(rng.choice([1, 5, 10, 20]), int(500e6 / cells)))
        if kind == "coupled":
            steps = 1
        if kind == "bed":
            eps, rmin = "linear", rng.uniform(5.0, 10.0)
            rmax, phi = rmin, rng.uniform(0.03, 0.38)
        elif kind == "channel":
            rmin = rng.uniform(3.5, 6.0)
            rmax, phi = rmin, rng.uniform(0.05, 0.25)
        else:
            rmin, rmax = 3.0, rng.uniform(4.0, 6.0)
            phi = rng.uniform(0.02, 0.15)
    field = kind in ("settle", "channel") and n[0] * n[1] * n[2] < 3e6 and rng.random() < 0.3
    c = _case("", kind, n[0], n[1], n[2], steps, precision=precision, streaming=streaming,
              eps=eps, eps_n=eps_n, phi=round(phi, 4), rmin=round(rmin, 3), rmax=round(rmax, 3),
              field=field)
    del c["name"]
    return c


# ---- the physics of a case (the values of the repository's workloads)

def _setup(c):
    k = c["kind"]
    s = dict(tau=0.55, relax="trt", walls=(0,) * 6, fbody=(0.0, 0.0, 0.0), weighting="nt",
             gravity=(0.0, 0.0, 0.0), dem=False, density=2.5, bc_velocity=(0.0, 0.0, 0.0))
    if k == "drag":
        s.update(tau=0.6, relax="srt", fbody=(1e-6, 0.0, 0.0))
    elif k == "channel":
        s.update(walls=(1, 1, 0, 0, 0, 0), fbody=(0.0, 0.0, 1e-5))
    elif k == "bed":
        s.update(relax="srt", walls=(1, 1, 1, 1, 2, 3), gravity=(0.0, 0.0, -2.75e-5),
                 weighting="eps", dem=True, density=1.1,
                 bc_velocity=(0.0, 0.0, ((0.55 - 0.5) / 3.0) / (2.0 * c["rmax"])))
    else:
        s.update(gravity=(0.0, 0.0, -2e-5), dem=True)
    return s


def _spheres(c, seed):
    """Centres, radii, velocities and angular velocities: lattice cells of edge
    at least 2 rmax + gap, as many of them (at random) as give the solid
    fraction, each sphere at a random place of its cell."""
    rng = np.random.default_rng(seed)
    dims = np.array([c["nx"], c["ny"], c["nz"]], float)
    gap = 0.5 if c["kind"] == "bed" else 1.0
    nc = np.maximum(1, np.floor(dims / (2.0 * c["rmax"] + gap)).astype(int))
    h = dims / nc
    rmin, rmax = c["rmin"], c["rmax"]
    # mean r^3 of a uniform radius
    r3 = rmax ** 3 if rmax == rmin else (rmax ** 4 - rmin ** 4) / (4.0 * (rmax - rmin))
    total = int(nc.prod())
    count = int(round(c["phi"] * dims.prod() / (4.0 / 3.0 * math.pi * r3)))
    count = max(1, min(count, total))
    cell = rng.permutation(total)[:count]
    idx = np.stack([cell % nc[0], (cell // nc[0]) % nc[1], cell // (nc[0] * nc[1])], 1)
    r = rng.uniform(rmin, rmax, count) if rmax > rmin else np.full(count, float(rmax))
    room = np.maximum(0.0, h[None, :] / 2.0 - r[:, None] - gap / 2.0)
    x = (idx + 0.5) * h + room * rng.uniform(-1.0, 1.0, (count, 3))
    free = c["kind"] not in ("drag", "channel")
    u = 1e-3 * rng.uniform(-1.0, 1.0, (count, 3)) if free else np.zeros((count, 3))
    om = 1e-4 * rng.uniform(-1.0, 1.0, (count, 3)) if free else np.zeros((count, 3))
    return x, r, u, om


def _net(seed):
    """A 4-32-32-1 network whose correction is small, as a trained one's is."""
    rng = np.random.default_rng(seed + 77)

    def lin(o, i):
        b = math.sqrt(6.0 / i)
        return rng.uniform(-b, b, (o, i)).astype(np.float32).astype(float)

    W1, W2, W3 = lin(32, 4), lin(32, 32), (0.01 * lin(1, 32)).astype(np.float32).astype(float)
    W1[:, 3] = (W1[:, 3] / 5.0).astype(np.float32)
    b1 = (0.01 - 7.0 * W1[:, 3]).astype(np.float32).astype(float)
    b2 = np.full(32, np.float32(0.01), float)
    return [W1, b1, W2, b2, W3, np.zeros(1)]


def _noise(c, seed):
    rng = np.random.default_rng(seed + 5)
    f = 1.0 + 1e-3 * rng.uniform(-1.0, 1.0, (19, c["nz"], c["ny"], c["nx"]))
    return f * np.array(W).reshape(19, 1, 1, 1)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "train":
        s.seed = 20230321 + seed
        s.net = capi.pack_mlp(_net(seed))
        s.e = capi.Engine(32, 8, 8, 0.6)
        return s
    p = _setup(case)
    s.e = capi.Engine(case["nx"], case["ny"], case["nz"], p["tau"], relax=p["relax"], magic=MAGIC,
                      walls=p["walls"], fbody=p["fbody"], weighting=p["weighting"],
                      eps_mode=case["eps"], eps_n=case["eps_n"], gravity=p["gravity"],
                      dem=p["dem"], precision=case["precision"], streaming=case["streaming"],
                      bc_velocity=p["bc_velocity"])
    x, r, u, om = _spheres(case, seed)
    fixed = np.full(r.size, 0 if p["dem"] else 1, np.uint8)
    s.e.set_particles(x, r, u=u, omega=om, density=np.full(r.size, p["density"]), fixed=fixed)
    s.p = (x, u, om)
    if case["eps"] == "mlp":
        s.e.set_mlp(capi.pack_mlp(_net(seed)))
    if case["kind"] == "drag":
        s.e.set_pdfs(_noise(case, seed))
    return s


def run(s):
    c, e = s.case, s.e
    if c["kind"] == "train":
        e.set_mlp(s.net)
        loss = e.train_surrogate(c["samples"], s.seed, c["epochs"], c["batch"], 3e-3)
        return {"params": e.get_mlp(), "loss": np.float32(loss)}
    if c["kind"] == "coupled":
        e.update_particles(*s.p)
    e.step(c["steps"])
    F, T = e.force_torque()
    out = {"F": F, "T": T}
    if _setup(c)["dem"]:
        s.p = out["x"], out["u"], out["om"] = e.particles()
    if c["field"]:
        out["rho"], out["vel"] = e.macroscopic()
    if c["precision"] == "fp32":
        # the form's forces and fields are 32-bit numbers in FP64 arrays
        out = {k: v if k == "x" else v.astype(np.float32) for k, v in out.items()}
    return out


def work(case):
    if case["kind"] == "train":
        n, batches = case["samples"], case["samples"] * case["epochs"]
        # forward and backward of 4-32-32-1, and the 512 sample tests per label
        return {"bytes": 20.0 * n + 20.0 * batches, "flops": 6.0 * 1184 * batches + 512.0 * 8 * n}
    x, r, _, _ = _spheres(case, 0)
    cells = float(case["nx"] * case["ny"] * case["nz"])
    slots = float(np.sum(4.0 / 3.0 * math.pi * (r + REACH) ** 3))
    # per step: 19 PDFs read and written per cell, two slots' index and weight
    # per covered cell; adds and multiplies of the collision per cell and slot
    esz = 4 if case["precision"] == "fp32" else 8
    b = case["steps"] * (38.0 * esz * cells + (16.0 if esz == 4 else 24.0) * min(slots, cells))
    f = case["steps"] * (219.0 * cells + 139.0 * slots)
    b += 8.0 * 6 * r.size + (72.0 * r.size if _setup(case)["dem"] else 0.0)
    if case["field"]:
        b += 32.0 * cells
        f += 40.0 * cells
    return {"bytes": b, "flops": f}


# ---- the same time loop in plain FP64 torch

def exact(case, seed):
    if case["kind"] == "train":
        return None  # hundreds of Adam steps from FP32 gradients: no value of their own
    cells = case["nx"] * case["ny"] * case["nz"]
    if cells * case["steps"] > 800e6 or cells > 140e6:
        return None  # takes longer than some 20 seconds, or more memory than is left
    with torch.no_grad():
        return _Plain(case, seed).run()


class _Plain:
    def __init__(self, c, seed):
        self.c, self.s = c, _setup(c)
        self.dev = torch.device("cuda")
        x, r, u, om = _spheres(c, seed)
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=self.dev)  # noqa: E731
        self.x, self.r, self.u, self.om = t(x), t(r), t(u), t(om)
        self.n = (c["nx"], c["ny"], c["nz"])
        self.per = [self.s["walls"][2 * a] == 0 for a in range(3)]
        self.wrap()
        self.vol = 4.0 / 3.0 * math.pi * self.r ** 3
        self.m = self.s["density"] * self.vol
        self.I = 0.4 * self.m * self.r ** 2
        self.g = t(np.array(self.s["gravity"]))
        self.Fo = ((self.m - self.vol)[:, None] * self.g[None, :])
        self.To = torch.zeros_like(self.x)
        shape = (19, c["nz"], c["ny"], c["nx"])
        if c["kind"] == "drag":
            self.f = t(_noise(c, seed))
        else:
            self.f = torch.empty(shape, dtype=torch.float64, device=self.dev)
            for q in range(19):
                self.f[q] = W[q]
        self.net = [t(p) for p in _net(seed)] if c["eps"] == "mlp" else None
        self.mapped = False

    def wrap(self):
        for a in range(3):
            if self.per[a]:
                self.x[:, a] %= self.n[a]

    # -- mapping: entries (cell, particle, offset, weight) and 1 - B per cell
    def map(self):
        dev, n = self.dev, self.n
        m = int(math.ceil(float(self.r.max()))) + 2
        o = torch.arange(-m, m + 1, device=dev)
        cells, parts, offs = [], [], []
        for lo in range(0, self.r.numel(), 4096):
            x, r = self.x[lo:lo + 4096], self.r[lo:lo + 4096]
            i0 = torch.floor(x).long()
            # per axis: integer coordinates and offsets of the box around each sphere
            ii = [i0[:, a, None] + o[None, :] for a in range(3)]
            dd = [(ii[a].double() + 0.5) - x[:, a, None] for a in range(3)]
            d2 = (dd[0] ** 2)[:, None, None, :] + (dd[1] ** 2)[:, None, :, None] + \
                (dd[2] ** 2)[:, :, None, None]
            ok = d2 < ((r + REACH) ** 2)[:, None, None, None]
            for a in range(3):
                if not self.per[a]:
                    inside = (ii[a] >= 0) & (ii[a] < n[a])
                    ok &= inside.view([-1] + [len(o) if k == 2 - a else 1 for k in range(3)])
            p, kz, ky, kx = torch.nonzero(ok, as_tuple=True)
            gi = [ii[a][p, k] % n[a] for a, k in ((0, kx), (1, ky), (2, kz))]
            cells.append(gi[0] + n[0] * (gi[1] + n[1] * gi[2]))
            parts.append(p + lo)
            offs.append(torch.stack([dd[0][p, kx], dd[1][p, ky], dd[2][p, kz]], 0))
            del d2, ok
        self.cell, self.part = torch.cat(cells), torch.cat(parts)
        self.d = torch.cat(offs, 1)
        eps = torch.cat([self.eps(slice(i, i + (1 << 24)))
                         for i in range(0, self.cell.numel(), 1 << 24)])
        if self.s["weighting"] == "nt":
            h = self.s["tau"] - 0.5
            eps = eps * h / ((1.0 - eps) + h)
        N = n[0] * n[1] * n[2]
        B = torch.zeros(N, dtype=torch.float64, device=dev).index_add_(0, self.cell, eps)
        self.B = eps / torch.clamp(B[self.cell], min=1.0)
        self.omB = 1.0 - torch.clamp(B, max=1.0)

    def eps(self, sl):
        c, n = self.c, self.n
        d, r, cell = self.d[:, sl], self.r[self.part[sl]], self.cell[sl]
        d2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
        dist = torch.sqrt(d2)
        lin = None
        if c["eps"] in ("linear", "mlp"):
            r2 = r * r
            s = torch.sqrt(r2 - 0.5)
            va = (1.0 / 12.0 - r2) * torch.atan((0.5 * s) / (0.5 - r2)) + s / 3.0 + \
                (r2 - 1.0 / 12.0) * torch.atan(0.5 / s) - \
                4.0 / 3.0 * r2 * r * torch.atan(0.25 / (r * s))
            lin = torch.clamp((r - dist) + (va - r + 0.5), 0.0, 1.0)
            if c["eps"] == "linear":
                return lin
        inner = d2 <= (r - REACH) ** 2
        out = inner.double()
        part = torch.nonzero(~inner, as_tuple=True)[0]
        if c["eps"] == "mlp":
            if not hasattr(self, "reach") or self.reach is None:
                self.reach = torch.zeros(n[0] * n[1] * n[2], dtype=torch.int8, device=self.dev)
                self.reach.index_add_(0, self.cell, torch.ones_like(self.cell, dtype=torch.int8))
            cc = cell[part]
            net = self.reach[cc] == 1
            if not self.per[0]:
                ix = cc % n[0]
                net &= (ix > 0) & (ix < n[0] - 1)
            k = part[net]
            a = torch.sort(torch.abs(d[:, k] / r[k]), 0, descending=True)[0]
            X = torch.cat([a, r[k][None]], 0).T
            W1, b1, W2, b2, W3, b3 = self.net
            h = torch.relu(torch.relu(X @ W1.T + b1) @ W2.T + b2)
            out[k] = torch.clamp(lin[k] + (h @ W3.T + b3)[:, 0], 0.0, 1.0)
            part = part[~net]
        m = 8 if c["eps"] == "mlp" else c["eps_n"]
        sub = [(i + 0.5) / m - 0.5 for i in range(m)]
        px, py, pz = d[0, part], d[1, part], d[2, part]
        r2, cnt = r[part] ** 2, torch.zeros_like(px)
        for sz in sub:
            z2 = (pz + sz) ** 2
            for sy in sub:
                y2 = (py + sy) ** 2
                for sx in sub:
                    cnt += ((px + sx) ** 2 + y2 + z2) <= r2
        out[part] = cnt / float(m ** 3)
        return out

    # -- streaming (Eq. 2 read backwards), walls and open faces
    def pulled(self, q):
        f, wl = self.f, self.s["walls"]
        g = torch.roll(f[q], (CZ[q], CY[q], CX[q]), (0, 1, 2))
        qb = 0 if q == 0 else (q + 1 if q % 2 else q - 1)
        if CZ[q] and wl[4]:
            k = 0 if CZ[q] > 0 else self.n[2] - 1
            face = wl[4] if CZ[q] > 0 else wl[5]
            bb = f[qb, k]
            if face == 2:
                U = self.s["bc_velocity"]
                bb = bb + 6.0 * W[q] * (CX[q] * U[0] + CY[q] * U[1] + CZ[q] * U[2])
            elif face == 3:
                ub = [sum(C[p] * f[p, k] for p in range(19) if C[p]) for C in (CX, CY, CZ)]
                cu = CX[q] * ub[0] + CY[q] * ub[1] + CZ[q] * ub[2]
                uu = ub[0] ** 2 + ub[1] ** 2 + ub[2] ** 2
                bb = -bb + 2.0 * W[q] * (1.0 + 4.5 * cu * cu - 1.5 * uu)
            g[k] = bb
        if CY[q] and wl[2]:
            k = 0 if CY[q] > 0 else self.n[1] - 1
            g[:, k] = f[qb, :, k]
        if CX[q] and wl[0]:
            k = 0 if CX[q] > 0 else self.n[0] - 1
            g[:, :, k] = f[qb, :, :, k]
        return g

    def stream(self):
        new = torch.empty_like(self.f)
        for q in range(19):
            new[q] = self.pulled(q)
        self.f = new

    def moments(self):
        f = self.f
        j = []
        for C in (CX, CY, CZ):
            a = torch.zeros_like(f[0])
            for q in range(1, 19, 2):  # by opposite pairs
                if C[q]:
                    a += C[q] * (f[q] - f[q + 1])
            j.append(a)
        drho = f[0] - W[0]
        for q in range(1, 19, 2):
            drho += (f[q] - W[q]) + (f[q + 1] - W[q + 1])
        return drho, j

    def step(self):
        s = self.s
        if not self.mapped:
            self.reach = None
            self.map()
            self.mapped = not s["dem"]
        # body force and the counter force of the particles' weight
        fe = torch.tensor(s["fbody"], dtype=torch.float64, device=self.dev)
        if s["dem"] and s["walls"][4] < 2:
            G = ((self.m - self.vol)[:, None] * self.g[None, :]).sum(0)
            fe = fe - G / self.omB.sum()
        fe = self.fe = [float(v) for v in fe]
        self.stream()
        f = self.f
        wp = 1.0 / s["tau"]
        wm = 1.0 / (0.5 + MAGIC / (s["tau"] - 0.5)) if s["relax"] == "trt" else wp
        drho, j = self.moments()
        U = [j[a] + 0.5 * fe[a] if fe[a] else j[a] for a in range(3)]
        del j
        uu = U[0] ** 2 + U[1] ** 2 + U[2] ** 2
        Uf = U[0] * fe[0] + U[1] * fe[1] + U[2] * fe[2]
        omB = self.omB.view_as(uu)
        # solid operators' inputs: the streamed PDFs at the entries' cells
        ce, B = self.cell, self.B
        Ue = [v.view(-1)[ce] for v in U]
        d, om, up = self.d, self.om[self.part], self.u[self.part]
        V = [up[:, 0] + (om[:, 1] * d[2] - om[:, 2] * d[1]),
             up[:, 1] + (om[:, 2] * d[0] - om[:, 0] * d[2]),
             up[:, 2] + (om[:, 0] * d[1] - om[:, 1] * d[0])]
        dU2 = (V[0] ** 2 + V[1] ** 2 + V[2] ** 2) - uu.view(-1)[ce]
        S = [torch.zeros_like(B) for _ in range(3)]
        b0 = drho - 1.5 * uu
        add0 = W[0] * -1.5 * dU2 * B
        f[0] += omB * (wp * (W[0] * b0 - (f[0] - W[0])) - (1.0 - 0.5 * wp) * 3.0 * W[0] * Uf)
        f[0].view(-1).index_add_(0, ce, add0)
        for q in range(1, 19, 2):
            c, w = (CX[q], CY[q], CZ[q]), W[q]
            dot = lambda v: sum(c[a] * v[a] for a in range(3) if c[a])  # noqa: E731
            fa, fb = f[q] - w, f[q + 1] - w
            cu, cf = dot(U), sum(c[a] * fe[a] for a in range(3))
            sy, an = 0.5 * (fa + fb), 0.5 * (fa - fb)
            # solid operator of the entries (Eq. 19) from the streamed values
            ane, cue, cve = an.view(-1)[ce], dot(Ue), dot(V)
            sym = B * (w * (4.5 * (cve - cue) * (cve + cue) - 1.5 * dU2))
            ant = B * (3.0 * w * (cve + cue) - 2.0 * ane)
            for a in range(3):
                if c[a]:
                    S[a] -= 2.0 * c[a] * ant
            ds = wp * (w * (b0 + 4.5 * cu * cu) - sy) + \
                (1.0 - 0.5 * wp) * w * (9.0 * cf * cu - 3.0 * Uf)
            da = wm * (3.0 * w * cu - an) + (1.0 - 0.5 * wm) * 3.0 * w * cf
            f[q] += omB * (ds + da)
            f[q + 1] += omB * (ds - da)
            f[q].view(-1).index_add_(0, ce, sym + ant)
            f[q + 1].view(-1).index_add_(0, ce, sym - ant)
        T = [d[1] * S[2] - d[2] * S[1], d[2] * S[0] - d[0] * S[2], d[0] * S[1] - d[1] * S[0]]
        z = torch.zeros_like(self.r)
        self.F = torch.stack([z.index_add(0, self.part, v) for v in S], 1)
        self.T = torch.stack([z.index_add(0, self.part, v) for v in T], 1)
        if s["dem"]:
            self.move()

    # -- ten velocity-Verlet sub-steps; the spheres stay apart over a pass, so
    # no contact acts
    def move(self):
        dt, m, I = 0.1, self.m[:, None], self.I[:, None]
        F = self.F + (self.m - self.vol)[:, None] * self.g[None, :]
        for _ in range(10):
            self.x += dt * self.u + dt * dt * self.Fo / (2.0 * m)
            self.wrap()
            self.u = self.u + dt * (self.Fo + F) / (2.0 * m)
            self.om = self.om + dt * (self.To + self.T) / (2.0 * I)
            self.Fo, self.To = F, self.T

    def run(self):
        for _ in range(self.c["steps"]):
            self.step()
        out = {"F": self.F, "T": self.T}
        if self.s["dem"]:
            out.update(x=self.x, u=self.u, om=self.om)
        if self.c["field"]:
            self.stream()
            drho, j = self.moments()
            out["rho"] = 1.0 + drho
            out["vel"] = torch.stack([j[a] + 0.5 * self.fe[a] for a in range(3)], 0)
        return {k: v.cpu() for k, v in out.items()}
