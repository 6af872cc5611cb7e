"""Performance cases of the plane-strain lattice Boltzmann solver.

Each case is one job as a user's program runs it through the Python binding:
initial displacements on the device, a number of time steps, fields read back
into device tensors.  The sizes, materials, edges and step counts are those of
``workloads.py``, of the tests and of ``bench.py`` (the step counts of the
long runs cut so that a pass stays well under a second).

``exact`` restates the method in FP64 torch operations on whole arrays: one
array operation per term of the scheme, boundary points through index lists.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2301_00228_gb300 import lbps
from paper_2301_00228_gb300 import workloads as W

N, D = W.NEUMANN, W.DIRICHLET
A0 = 0.9999
FIELDS = ("ux", "uy", "vx", "vy", "phi", "psi")
EDGES = {  # edge types in the order bottom, right, top, left
    "left": (N, N, N, D),       # the 64 x 64 square
    "bottom": (D, N, N, N),     # the many-pulse plate
    "mixed": None,              # drawn from the seed, with edge values, as the batches and requests
    "free": (N, N, N, N),       # the tension examples
}


def listed():
    return [
        # the plain method in FP64: the 64 x 64 square with a clamped edge
        dict(name="square_64_f64", kind="solve", nx=64, ny=64, storage="f64", edges="left", steps=1000),
        # a program that looks at the lattice after every step: one call, one step
        dict(name="stepwise_128x96_f32", kind="stepwise", nx=128, ny=96, storage="f32", edges="mixed", steps=200),
        # the tension square: ramped traction, synchronised every 50 steps
        dict(name="tension_256_f32", kind="tension", nx=256, ny=256, storage="f32", edges="free", steps=1000),
        # one request of the serving stream: ragged sides, random edges and material
        dict(name="request_389x1171_f32", kind="solve", nx=389, ny=1171, storage="f32", edges="mixed", steps=1000),
        # a solve whose energy is recorded as it runs
        dict(name="monitored_700x500_f32", kind="monitored", nx=700, ny=500, storage="f32", edges="bottom",
             steps=500, every=25),
        # plane waves on a periodic lattice
        dict(name="waves_1024_f32", kind="waves", nx=1024, ny=1024, storage="f32", edges="free", steps=500),
        # the plate with a hole: general geometry, ramped traction, synchronisation
        dict(name="hole_1024_f32", kind="hole", nx=1024, ny=1024, storage="f32", edges="free", steps=400),
        # the size of the precision crop, BF16 pair sums
        dict(name="crop_1024_bf16", kind="solve", nx=1024, ny=1024, storage="bf16", edges="bottom", steps=400),
        # 256 uneven lattices in one batch, two steps per sweep as the server runs them
        dict(name="batch_256_f32", kind="batch", nx=512, ny=512, storage="f32", edges="mixed", steps=400, count=256),
        # a large request, odd sides, FP16 pair sums
        dict(name="request_2047x1533_f16", kind="solve", nx=2047, ny=1533, storage="f16", edges="mixed", steps=300),
        # a quarter of the largest plate, BFP13 pair sums
        dict(name="pulses_4096_bfp13", kind="solve", nx=4096, ny=4096, storage="bfp13", edges="bottom", steps=200),
        # the many-pulse plate in full
        dict(name="pulses_8192_f32", kind="solve", nx=8192, ny=8192, storage="f32", edges="bottom", steps=100),
    ]


def draw(rng):
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve"] * 6 + ["stepwise", "tension", "monitored", "waves", "hole", "batch"])
    storage = "f32"
    edges = "free"
    case = {}
    if kind == "solve":
        nx, ny = side(64, 6144), side(64, 6144)
        storage = rng.choice(["f32", "f32", "f16", "bf16", "bfp13"] + (["f64"] if nx * ny <= 1 << 18 else []))
        edges = rng.choice(["mixed", "bottom", "left"])
    elif kind == "batch":
        nx = ny = 512
        case["count"] = rng.randint(16, 256)
        edges = "mixed"
    elif kind == "stepwise":
        nx, ny = side(32, 1024), side(32, 1024)
        edges = "mixed"
    elif kind == "monitored":
        nx, ny = side(128, 2048), side(128, 2048)
        storage = rng.choice(["f32", "f16", "bfp13"])
        edges = rng.choice(["mixed", "bottom"])
    elif kind == "waves":
        nx = ny = side(256, 2048)
        storage = rng.choice(["f32", "bfp13"])
    elif kind == "tension":
        nx = ny = side(64, 1024)
    else:
        nx = ny = side(128, 2048)
        storage = rng.choice(["f32", "bfp13"])
    points = nx * ny * case.get("count", 1) // (3 if kind == "batch" else 1)
    most = int(min(1000, 3_000_000_000 // points))
    steps = max(50, rng.randint(most // 2, most))
    if kind == "stepwise":
        steps = rng.randint(50, 300)
    if kind == "monitored":
        case["every"] = rng.choice([10, 25, 40])
        steps = max(1, steps // case["every"]) * case["every"]
    return dict(kind=kind, nx=nx, ny=ny, storage=storage, edges=edges, steps=steps, **case)


# ------------------------------------------------------------------ inputs

def _domain(case, seed):
    """The problem of one lattice, from the seed alone."""
    rng = np.random.default_rng([seed, case["nx"], case["ny"]])
    nx, ny, kind = case["nx"], case["ny"], case["kind"]
    if kind in ("tension", "hole"):
        d = (W.tension_square if kind == "tension" else W.hole_square)(nx, a0_phi=A0)
        # the paper's amplitude 0.005 mu is one choice of a user's load
        amp = rng.uniform(0.5, 1.5)
        d.edge_value = tuple((amp * x, amp * y) for x, y in d.edge_value)
        return d
    if kind == "waves":
        m, n = W.pick_wave_numbers(nx, 64.0, rng)
        return W.Domain(nx, ny, 2.0, 1.0, a0_phi=A0, periodic_x=True, periodic_y=True,
                        wave=(m, n, float(rng.uniform(5e-4, 2e-3)), float(rng.uniform(5e-4, 2e-3))))
    if case["edges"] == "mixed":
        et = tuple(int(x) for x in rng.choice([N, D], size=4))
        ev = tuple((float(a), float(b)) for a, b in rng.uniform(-1e-3, 1e-3, size=(4, 2)))
        lam = float(rng.uniform(0.5, 4.0))
    else:
        et, ev, lam = EDGES[case["edges"]], ((0.0, 0.0),) * 4, 3.0 if case["edges"] == "bottom" else 1.0
    pulses = []
    for _ in range(max(1, min(32, nx * ny >> 19))):
        sg = float(rng.uniform(min(4.0, nx / 12), max(5.0, min(64.0, min(nx, ny) / 12))))
        pulses.append((float(rng.uniform(0, nx - 1)), float(rng.uniform(0, ny - 1)), sg, 1e-3,
                       "dilatation" if rng.random() < 0.5 else "rotation"))
    return W.Domain(nx, ny, lam, 1.0, a0_phi=A0, edge_type=et, edge_value=ev, pulses=pulses)


def _domains(case, seed):
    if case["kind"] != "batch":
        return [_domain(case, seed)]
    # the sizes belong to the case, everything else to the seed
    sizes = np.random.default_rng(case["count"]).integers(64, 513, size=(case["count"], 2))
    rng = np.random.default_rng([seed, case["count"]])
    doms = []
    for nx, ny in sizes.tolist():
        d = W.random_rectangle(rng)
        _, _, sigma, amp, pulse = d.pulses[0]
        at = (float(rng.integers(0, nx)), float(rng.integers(0, ny)))
        doms.append(W.Domain(nx, ny, d.lam, d.mu, a0_phi=A0, edge_type=d.edge_type, edge_value=d.edge_value,
                             pulses=[(*at, sigma, amp, pulse)]))
    return doms


def _lattice(case, d):
    sync = 50 if case["kind"] in ("tension", "hole") else 0
    et, ev = d.edge_arrays()
    kw = dict(rho=d.rho, a0_phi=d.a0_phi, storage=case["storage"], sync_every=sync)
    if d.hole is not None:
        nt, bv, cell = lbps.lbps_disk_cells(d.nx, d.ny, 1.0, *d.hole, et, ev)
        lat = lbps.Lattice(d.nx, d.ny, d.lam, d.mu, node_type=nt, bc_value=bv, cell=cell, **kw)
    elif d.periodic_x:
        lat = lbps.Lattice(d.nx, d.ny, d.lam, d.mu, periodic_x=True, periodic_y=True, **kw)
    else:
        lat = lbps.Lattice.rectangle(d.nx, d.ny, d.lam, d.mu, et, ev, **kw)
    for load_kind, ramp, hold in d.loads:
        lat.set_load(load_kind, ramp, hold)
    return lat


def prepare(case, seed):
    """The lattice (or batch), the initial displacements and the tensors the
    fields are read into."""
    doms = _domains(case, seed)
    state = dict(case=case, lats=[_lattice(case, d) for d in doms],
                 u0=[d.displacement_torch() for d in doms])
    total = sum(d.nx * d.ny for d in doms)
    state["out"] = {k: torch.empty(total, dtype=torch.float64, device="cuda") for k in FIELDS}
    at, views = 0, []
    for d in doms:
        views.append({k: v[at:at + d.nx * d.ny].view(1, d.ny, d.nx) for k, v in state["out"].items()})
        at += d.nx * d.ny
    state["views"] = views
    if case["kind"] == "batch":
        for lat, u in zip(state["lats"], state["u0"]):
            lat.init(*u)
        state["batch"] = lbps.Batch(state["lats"], stream=torch.cuda.current_stream())
        state["batch"].set_step_pairs(True)
    return state


# --------------------------------------------------------------- one pass

def run(state):
    """One solve: initialise, step, read the fields."""
    case = state["case"]
    for lat, u in zip(state["lats"], state["u0"]):
        lat.init(*u)
    lat, energy = state["lats"][0], []
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
    elif case["kind"] == "stepwise":
        for _ in range(case["steps"]):
            lat.step(1)
    elif case["kind"] == "monitored":
        for _ in range(case["steps"] // case["every"]):
            lat.step(case["every"])
            energy.append(lat.energy())
    else:
        lat.step(case["steps"])
    for lat, views in zip(state["lats"], state["views"]):
        for k, v in views.items():
            lat.read_device(k, out=v)
    out = dict(state["out"])
    if energy:
        out["energy"] = np.stack(energy)
    return out


def work(case):
    """What a solve cannot do without: u(x, 0) read and the fields written
    once, and per point and time step the operations of the scheme (the
    moments, the equilibria and the streamed populations of both sets, the
    acceleration, the integration of u: about 90)."""
    points = case["nx"] * case["ny"]
    if case["kind"] == "batch":
        points = case["count"] * 288 * 288  # sides U{64..512}
    return {"bytes": points * 8 * (2 + len(FIELDS)), "flops": 90.0 * points * case["steps"]}


# ------------------------------------------------- the method in 64 bits

def _disk_area(x0, x1, y0, y1, r):
    """Area of [x0, x1] x [y0, y1] inside the disk of radius r at the origin
    (arrays): the chord integrated piece by piece between the points where it
    meets the horizontal sides or ends."""
    cuts = [x0, x1]
    for y in (y0, y1):
        h = np.sqrt(np.maximum(r * r - y * y, 0.0))
        cuts += [np.clip(h, x0, x1), np.clip(-h, x0, x1)]
    cuts += [np.clip(r, x0, x1), np.clip(-r, x0, x1)]
    cuts = np.sort(np.stack(cuts), axis=0)

    def H(x):  # antiderivative of the half chord
        t = np.clip(x / r, -1.0, 1.0)
        return 0.5 * r * r * (t * np.sqrt(1.0 - t * t) + np.arcsin(t))

    area = np.zeros_like(x0)
    for a, b in zip(cuts[:-1], cuts[1:]):
        m = 0.5 * (a + b)
        h = np.sqrt(np.maximum(r * r - m * m, 0.0))
        chord = H(b) - H(a)
        top = np.where(h < y1, chord, y1 * (b - a))
        bot = np.where(-h > y0, -chord, y0 * (b - a))
        inside = (np.abs(m) < r) & (np.minimum(h, y1) > np.maximum(-h, y0)) & (b > a)
        area += np.where(inside, top - bot, 0.0)
    return area


class _Exact:
    """The scheme on one array of points: types 0 interior, 1 Neumann, 2
    Dirichlet, 3 outside the body; material constants per row, so that many
    lattices may lie one above the other in it."""

    def __init__(self, types, force, lam, mu, rho, a0, px=False, py=False, hole=None, ramp=None, sync=0):
        dev = "cuda"
        ny, nx = types.shape
        self.shape, self.per, self.sync, self.ramp, self.steps = (ny, nx), (px, py), sync, ramp, 0
        self.lam, self.mu, self.rho = lam, mu, rho
        self.cd2, self.cs2 = (lam + 2 * mu) / rho, mu / rho
        self.a = torch.stack([(1 - a0) / 4 + 0 * mu, self.cs2 / self.cd2 * (1 - a0) / 4])   # [set, rows, 1]
        self.dt = torch.sqrt(2 * self.a[0]) / torch.sqrt(self.cd2)
        body = types != 3
        self.body, self.inner = body, types == 0
        # a point's neighbours in the directions E, N, W, S: linear index, and whether it is in the body
        J, I = torch.nonzero(body & (types != 0), as_tuple=True)
        self.type = types[J, I]
        self.k = J * nx + I

        def look(i, j):
            ok = torch.ones_like(i, dtype=torch.bool)
            if not px:
                ok &= (i >= 0) & (i < nx)
            if not py:
                ok &= (j >= 0) & (j < ny)
            i, j = i % nx, j % ny
            return ok & body[j, i], j * nx + i

        def stencil(i, j):
            """Second-order differences at the points (i, j): per axis the
            linear indices and weights of three points."""
            out = []
            for dx, dy in ((1, 0), (0, 1)):
                hp, kp = look(i + dx, j + dy)
                hm, km = look(i - dx, j - dy)
                _, kp2 = look(i + 2 * dx, j + 2 * dy)
                _, km2 = look(i - 2 * dx, j - 2 * dy)
                k0 = j * nx + i
                mid = (hp & hm)[:, None]
                fwd = hp[:, None]
                idx = torch.where(mid, torch.stack([km, kp, k0], 1),
                                  torch.where(fwd, torch.stack([k0, kp, kp2], 1), torch.stack([k0, km, km2], 1)))
                w = torch.tensor([[-0.5, 0.5, 0.0], [-1.5, 2.0, -0.5], [1.5, -2.0, 0.5]], dtype=torch.float64,
                                 device=dev)
                sel = torch.where(mid[:, 0], 0, torch.where(fwd[:, 0], 1, 2))
                out.append((idx, w[sel]))
            return out

        self.at_b = stencil(I, J)
        has, near = [], []
        for dx, dy in ((1, 0), (0, 1), (-1, 0), (0, -1)):
            h, _ = look(I + dx, J + dy)
            has.append(h)
            near.append((stencil(torch.where(h, I + dx, I) % nx, torch.where(h, J + dy, J) % ny)))
        self.near = near
        # cells: the square of side 1 clipped where neighbours are missing ...
        wx = 0.5 * has[0] + 0.5 * has[2]
        wy = 0.5 * has[1] + 0.5 * has[3]
        vol = wx * wy
        side = [torch.where(h, s, 0.0 * s) for h, s in zip(has, (wy, wx, wy, wx))]
        if hole is not None:  # ... and, around the hole, the square less the disk
            cx, cy, r = hole
            x, y = I.cpu().numpy() - cx, J.cpu().numpy() - cy
            ring = np.hypot(x, y) < r + 2.0
            ins = _disk_area(x - 0.5, x + 0.5, y - 0.5, y + 0.5, r)

            def left(c, o):  # of a unit side at distance c from the centre, along o +- 1/2: the part outside
                h = np.sqrt(np.maximum(r * r - c * c, 0.0))
                return 1.0 - np.maximum(0.0, np.minimum(o + 0.5, h) - np.maximum(o - 0.5, -h))

            sides = [left(x + 0.5, y), left(y + 0.5, x), left(x - 0.5, y), left(y - 0.5, x)]
            on = torch.from_numpy(ring).to(dev)
            vol = torch.where(on, torch.from_numpy(1.0 - ins).to(dev), vol)
            side = [torch.where(on, torch.from_numpy(s).to(dev), o) for s, o in zip(sides, side)]
        self.side = side
        row = J
        self.row = row
        self.inv_m = 1.0 / (rho[row, 0] * torch.where(vol > 0, vol, torch.ones_like(vol)))
        self.force = force[J, I].T.contiguous()
        self.f = torch.zeros((2, 5, ny, nx), dtype=torch.float64, device=dev)
        self.u = torch.zeros((4, ny, nx), dtype=torch.float64, device=dev)

    # differences at listed points and over the array
    @staticmethod
    def _diff(g, st):
        idx, w = st
        return (g.reshape(-1)[idx] * w).sum(1)

    def _grad(self, g):
        gx = (torch.roll(g, -1, 1) - torch.roll(g, 1, 1)) * 0.5
        gy = (torch.roll(g, -1, 0) - torch.roll(g, 1, 0)) * 0.5
        for out, st in zip((gx, gy), self.at_b):
            out.view(-1)[self.k] = self._diff(g, st)
        return gx, gy

    def _equilibrium(self, s, jx, jy, a):
        return torch.stack([(1 - 4 * a) * s, a * s + 0.5 * jx, a * s + 0.5 * jy, a * s - 0.5 * jx, a * s - 0.5 * jy])

    def _from_u(self, moments):
        """Populations at equilibrium with phi, psi from u and the given first moments."""
        (uxx, uxy), (uyx, uyy) = self._grad(self.u[0]), self._grad(self.u[1])
        for q, s in enumerate((uxx + uyy, uyx - uxy)):
            self.f[q] = self._equilibrium(s, *moments[q], self.a[q]) * self.body

    def init(self, ux, uy):
        self.u[0], self.u[1] = ux * self.body, uy * self.body
        zero = torch.zeros_like(ux)
        self._from_u([(zero, zero)] * 2)
        return self

    def _stress(self, st):
        exx, eyx = self._diff(self.u[0], st[0]), self._diff(self.u[1], st[0])
        exy, eyy = self._diff(self.u[0], st[1]), self._diff(self.u[1], st[1])
        lam, mu = self.lam[self.row, 0], self.mu[self.row, 0]
        tr = lam * (exx + eyy)
        return tr + 2 * mu * exx, tr + 2 * mu * eyy, mu * (exy + eyx)

    def _edge_acceleration(self):
        dt = self.dt[self.row, 0]
        ux, uy, vx, vy = (q.reshape(-1)[self.k] for q in self.u)
        fx, fy = self.force
        if self.ramp is not None:  # Neumann data, taken at the start of the step
            now = self.steps * dt
            scale = torch.clamp(now, max=self.ramp[1]) / self.ramp[0]
            fx, fy = fx * scale, fy * scale
        dir_x = 2 / dt ** 2 * (self.force[0] - ux) - 2 / dt * vx
        dir_y = 2 / dt ** 2 * (self.force[1] - uy) - 2 / dt * vy
        own = self._stress(self.at_b)
        for (nx, ny), length, st in zip(((1, 0), (0, 1), (-1, 0), (0, -1)), self.side, self.near):
            sxx, syy, sxy = (0.5 * (p + q) for p, q in zip(own, self._stress(st)))
            fx = fx + (sxx * nx + sxy * ny) * length
            fy = fy + (sxy * nx + syy * ny) * length
        fixed = self.type == D
        return torch.where(fixed, dir_x, fx * self.inv_m), torch.where(fixed, dir_y, fy * self.inv_m)

    def step(self):
        f, k, a, dt = self.f, self.k, self.a, self.dt
        s = f.sum(1)
        acc = torch.zeros_like(self.u[:2])
        (px, py), (qx, qy) = ((torch.roll(g, -1, 1) - torch.roll(g, 1, 1), torch.roll(g, -1, 0) - torch.roll(g, 1, 0))
                              for g in s)
        acc[0] = 0.5 * (self.cd2 * px - self.cs2 * qy)
        acc[1] = 0.5 * (self.cd2 * py + self.cs2 * qx)
        del px, py, qx, qy
        acc *= self.inner
        ex, ey = self._edge_acceleration()
        acc[0].view(-1)[k], acc[1].view(-1)[k] = ex, ey
        self.u[:2] += dt * self.u[2:] + 0.5 * dt ** 2 * acc
        self.u[2:] += dt * acc
        del acc
        # boundary points: populations with phi, psi of the new u
        (uxx, uxy), (uyx, uyy) = [[self._diff(self.u[q], st) for st in self.at_b] for q in (0, 1)]
        new = torch.zeros_like(f)
        OPP = (0, 3, 4, 1, 2)
        for q, sb in enumerate((uxx + uyy, uyx - uxy)):
            old = f[q].reshape(5, -1)[:, k]
            ab = a[q][self.row, 0]
            reset = self._equilibrium(sb, old[1] - old[3], old[2] - old[4], ab)
            mean = 0.5 * (old + reset)
            for al in range(5):
                w = (1 - 4 * a[q]) if al == 0 else a[q]
                out = 2 * w * s[q] - f[q, OPP[al]]
                if al:  # what boundary points send: the time-averaged state
                    out.view(-1)[k] = 2 * ab * mean.sum(0) - mean[OPP[al]]
                    out = torch.roll(out, 1 if al in (1, 2) else -1, 1 if al in (1, 3) else 0)
                new[q, al] = out * self.inner
                new[q, al].view(-1)[k] = reset[al]
        self.f = new
        self.steps += 1
        if self.sync and self.steps % self.sync == 0:
            self._from_u([(g[1] - g[3], g[2] - g[4]) for g in self.f.clone()])

    def energy(self):
        (uxx, uxy), (uyx, uyy) = self._grad(self.u[0]), self._grad(self.u[1])
        kin = (0.5 * self.rho * (self.u[2] ** 2 + self.u[3] ** 2) * self.body).sum()
        exy = 0.5 * (uxy + uyx)
        den = 0.5 * self.lam * (uxx + uyy) ** 2 + self.mu * (uxx ** 2 + uyy ** 2 + 2 * exy ** 2)
        strain = (den * self.body).sum()
        return [float(kin), float(strain), float(kin + strain)]

    def fields(self):
        s = self.f.sum(1)
        return dict(zip(FIELDS, (*self.u, *s)))


def _types(d, nt, force):
    """Node types and boundary data of one rectangle into nt [ny, nx] and
    force [ny, nx, 2]: u* at Dirichlet points (the mean where two edges meet),
    traction times the length of the outer faces at Neumann points."""
    ny, nx = nt.shape
    nt[:] = 0
    if d.periodic_x:
        return
    on = torch.zeros((4, ny, nx), dtype=torch.bool, device=nt.device)
    on[0, 0], on[1, :, -1], on[2, -1], on[3, :, 0] = True, True, True, True
    fixed = torch.tensor([t == D for t in d.edge_type], device=nt.device)[:, None, None]
    value = torch.tensor(d.edge_value, dtype=torch.float64, device=nt.device)[:, None, None, :]
    n_fixed, n_on = (on & fixed).sum(0), on.sum(0)
    nt[n_on > 0] = N
    nt[n_fixed > 0] = D
    target = ((on & fixed)[..., None] * value).sum(0) / n_fixed.clamp(min=1)[..., None]
    load = (on[..., None] * value).sum(0) * torch.where(n_on == 2, 0.5, 1.0)[..., None]
    force[:] = torch.where((n_fixed > 0)[..., None], target, load)


def exact(case, seed):
    doms = _domains(case, seed)
    # the lattices one above the other, a row outside the body between them
    rows, cols = sum(d.ny + 1 for d in doms) - 1, max(d.nx for d in doms)
    nt = torch.full((rows, cols), 3, dtype=torch.uint8, device="cuda")
    force = torch.zeros((rows, cols, 2), dtype=torch.float64, device="cuda")
    mat = torch.ones((4, rows, 1), dtype=torch.float64, device="cuda")
    ux = torch.zeros((rows, cols), dtype=torch.float64, device="cuda")
    uy = torch.zeros_like(ux)
    at, places = 0, []
    for d in doms:
        sl = slice(at, at + d.ny)
        places.append((sl, slice(0, d.nx)))
        _types(d, nt[sl, :d.nx], force[sl, :d.nx])
        if d.hole is not None:
            x = torch.arange(d.nx, dtype=torch.float64, device="cuda")
            void = (x[None, :] - d.hole[0]) ** 2 + (x[:, None] - d.hole[1]) ** 2 < d.hole[2] ** 2
            ring = torch.zeros_like(void)
            for ax in (0, 1):
                ring |= torch.roll(void, 1, ax) | torch.roll(void, -1, ax)
            nt[ring & ~void] = N
            nt[void] = 3
        for q, v in enumerate((d.lam, d.mu, d.rho, d.a0_phi)):
            mat[q, sl] = v
        ux[sl, :d.nx], uy[sl, :d.nx] = d.displacement_torch()
        at += d.ny + 1
    d = doms[0]
    sim = _Exact(nt, force, *mat, px=d.periodic_x, py=d.periodic_y, hole=d.hole,
                 ramp=d.loads[0][1:] if d.loads else None,
                 sync=50 if case["kind"] in ("tension", "hole") else 0).init(ux, uy)
    del ux, uy, nt, force
    energy = []
    for n in range(case["steps"]):
        sim.step()
        if case["kind"] == "monitored" and (n + 1) % case["every"] == 0:
            energy.append(sim.energy())
    out = {k: torch.cat([v[place].reshape(-1) for place in places]) for k, v in sim.fields().items()}
    if energy:
        out["energy"] = np.array(energy)
    return out
