"""The workloads whose speed counts: what a user of this package has it do, through its public classes.

A case is one stretch of time steps (or one gradient) and the result that a program then
takes from the device. Kinds:

  channel   one walled 2-D lattice with a steady porous void fraction: ``Lattice.step(n)``,
            then the populations (and, where ``macros`` is set, rho, u and p)
  moving    one periodic 2-D lattice whose void fraction and body force change every step,
            each handed over from device arrays before ``Lattice.step(1)``
  cube      one walled 3-D lattice: ``Lattice3D.step(n)``, then the populations (and rho, u, p)
  batch     many periodic lattices of mixed sizes advanced together: ``Batch.step(n)``, then
            every lattice's populations
  gradient  ``outlet_momentum``: the objective and its gradient in every cell

Lattices that store FP32, FP16 or BF16 hand their FP64 read-back on as FP32, as a program
does that keeps no more digits than the lattice holds. ``exact`` restates the scheme in
plain torch in 64 bits: D2Q9 (Eq. 5-7, 10, 13-20), its D3Q19 form, and torch's own
reverse mode for the gradient.
"""
import math
import random

import torch

import paper_2409_02964_gb300 as P

_DEV = "cuda" if torch.cuda.is_available() else "cpu"
_F64 = torch.float64
_SIZE = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}


def listed():
    return [
        # the manufactured solution on its own 64^2 lattice in FP64: phi, phi(t+1) and the
        # force handed over before each step, the smallest calls a study makes
        dict(name="moving64_fp64", kind="moving", n=64, storage="fp64", steps=20),
        # a small channel with odd sides, the sort a parameter sweep runs by the thousand
        dict(name="channel70_fp32", kind="channel", nx=130, ny=71, storage="fp32", steps=100, macros=True),
        # the 512^2 channel of the precision study
        dict(name="channel512_fp32", kind="channel", nx=512, ny=512, storage="fp32", steps=100),
        # the benchmark's 4096^2 channel, FP32, with the fields a run writes out
        dict(name="channel4096_fp32", kind="channel", nx=4096, ny=4096, storage="fp32", steps=64, macros=True),
        # the same flow with FP16 populations, on a ragged size
        dict(name="channel3000_fp16", kind="channel", nx=4001, ny=3001, storage="fp16", steps=64),
        # BF16 populations at a middling size
        dict(name="channel1200_bf16", kind="channel", nx=1200, ny=900, storage="bf16", steps=100),
        # the FP64 form that reference runs use
        dict(name="channel1024_fp64", kind="channel", nx=1024, ny=768, storage="fp64", steps=32),
        # flow around impermeable cells
        dict(name="solid1500_fp32", kind="channel", nx=1531, ny=1024, storage="fp32", steps=64, solid=True),
        # the 3-D channel of the benchmark
        dict(name="cube256_fp32", kind="cube", nx=256, ny=256, nz=256, storage="fp32", steps=10),
        # a small 3-D channel with ragged sides, and its FP64 form
        dict(name="cube48_fp64", kind="cube", nx=57, ny=48, nz=39, storage="fp64", steps=20, macros=True),
        # a batch of manufactured-solution lattices of mixed sizes
        dict(name="batch24_fp32", kind="batch", count=24, mix=5, storage="fp32", steps=32),
        # a design gradient on a small channel
        dict(name="gradient256_fp64", kind="gradient", nx=256, ny=192, nsteps=80, avg=20, every=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel", "channel", "channel", "cube", "cube", "moving", "batch", "gradient"])
    if kind == "channel":
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16", "fp64"])
        extra = rng.choice(["", "", "macros", "drag", "solid", "momentum"])
        if extra == "momentum" and storage not in ("fp16", "bf16"):
            extra = "macros"
        top = 900 if storage == "fp64" else 3000 if extra else 4000
        c = dict(kind=kind, nx=_log(rng, 24, top), ny=_log(rng, 16, top), storage=storage,
                 steps=rng.randint(8, 24) if storage == "fp64" else rng.randint(16, 64))
        if extra:
            c[extra] = True
        return c
    if kind == "cube":
        storage = rng.choice(["fp32", "fp32", "fp64"])
        top = 80 if storage == "fp64" else 240
        return dict(kind=kind, nx=_log(rng, 12, top), ny=_log(rng, 12, top), nz=_log(rng, 12, top), storage=storage,
                    steps=rng.randint(3, 10), macros=rng.random() < 0.3)
    if kind == "moving":
        return dict(kind=kind, n=_log(rng, 32, 160), storage=rng.choice(["fp64", "fp32", "fp32", "fp16"]),
                    steps=rng.randint(4, 24))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(6, 40), mix=rng.randint(0, 10 ** 6),
                    storage=rng.choice(["fp32", "fp32", "fp16", "bf16"]), steps=rng.randint(8, 32))
    nsteps = rng.randint(12, 80)
    return dict(kind=kind, nx=_log(rng, 24, 250), ny=_log(rng, 16, 190), nsteps=nsteps, avg=rng.randint(1, nsteps),
                every=rng.randint(4, 40))


# ---------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(seed))
    return g


def _smooth(shape, g, corr):
    """A periodic Gaussian random field (white noise filtered by exp(-|k|^2 l^2 / 2)), scaled to [0, 1]."""
    noise = torch.randn(shape, generator=g, device=_DEV, dtype=torch.float32).double()
    spec = torch.fft.rfftn(noise)
    for ax, n in enumerate(shape):
        k = 2.0 * math.pi * (torch.fft.rfftfreq(n) if ax == len(shape) - 1 else torch.fft.fftfreq(n)).to(_DEV, _F64)
        spec *= torch.exp(-0.5 * (k * corr) ** 2).reshape([-1 if a == ax else 1 for a in range(len(shape))])
    f = torch.fft.irfftn(spec, s=shape)
    return (f - f.min()) / (f.max() - f.min())


def _porous(shape, g):
    """The porous void fraction of the channels: random in [0.35, 1], a block of 0.4 with a
    ramp of two cells and a collar of 1 around it; float values, as FP32 lattices hold it."""
    phi = 0.35 + 0.65 * _smooth(shape, g, min(32.0, min(shape) / 8.0))
    depth = None
    for ax, n in enumerate(shape):
        a, b = int(round(0.4 * n)), int(round(0.6 * n))
        i = torch.arange(n, device=_DEV)
        d = torch.minimum(i - a, b - 1 - i).reshape([-1 if q == ax else 1 for q in range(len(shape))])
        depth = d if depth is None else torch.minimum(depth, d)
    collar = max(1, min(16, min(shape) // 16))
    phi = torch.where((depth < 0) & (depth >= -collar), torch.ones_like(phi), phi)
    for d in range(2):
        phi = torch.where(depth == d, torch.full_like(phi, 1.0 - 0.2 * (d + 1)), phi)
    phi = torch.where(depth >= 2, torch.full_like(phi, 0.4), phi)
    return phi.float().double().clamp(max=1.0)


def _solids(phi, g):
    """Impermeable cells: a block and a sprinkle of single cells."""
    ny, nx = phi.shape
    s = torch.rand(phi.shape, generator=g, device=_DEV) < 2e-4
    s[int(0.3 * ny):int(0.5 * ny), int(0.2 * nx):int(0.35 * nx)] = True
    return torch.where(s, torch.zeros_like(phi), phi)


def _gravity(ny):
    """The channels' drive along x: 1e-6, less in a wide one (it settles below u = 0.02)."""
    return min(1e-6, 8.0 * (0.1 / 3.0) * 0.02 / (ny * ny))


def _channel_inputs(c, seed):
    g = _gen(seed)
    ny, nx = c["ny"], c["nx"]
    phi = _porous((ny, nx), g)
    if c.get("solid"):
        phi = _solids(phi, g)
    corr = min(32.0, min(nx, ny) / 8.0)
    fluid = (phi > 0).double()
    u = [(0.02 * (_smooth((ny, nx), g, corr) - 0.5)).float().double() * fluid for _ in range(2)]
    return phi, torch.ones_like(phi), u


def _cube_inputs(c, seed):
    g = _gen(seed)
    shape = (c["nz"], c["ny"], c["nx"])
    phi = _porous(shape, g)
    u = torch.stack([(0.02 * (_smooth(shape, g, min(16.0, min(shape) / 6.0)) - 0.5)).float().double()
                     for _ in range(3)])
    return phi, torch.ones_like(phi), u


def _trig(terms, k, sx, cx, sy, cy):
    """A sum of coef * X(kx) * Y(ky), X and Y sine or cosine, and its derivatives to second order: {"", "x", "y", "xx", "xy", "yy"}."""
    def d(f):          # derivative of sine / cosine: (factor, function)
        return (k, "c") if f == "s" else (-k, "s")

    out = {}
    for name in ("", "x", "y", "xx", "xy", "yy"):
        acc = 0.0
        for coef, fx, fy in terms:
            m = coef
            for ax in name:
                if ax == "x":
                    q, fx = d(fx)
                else:
                    q, fy = d(fy)
                m = m * q
            acc = acc + m * (sx if fx == "s" else cx) * (sy if fy == "s" else cy)
        out[name] = acc
    return out


def _manufactured(n, t, tau, amp, period, u0, phi0=0.7):
    """phi, u and the body force (the momentum residual at rho = 1 without the pressure term)
    of phi = phi0 + A sin kx sin ky cos wt, phi u = grad psi + rot Psi, at the steps t (a tensor)."""
    k, w, nu = 2.0 * math.pi / n, 2.0 * math.pi / period, (tau - 0.5) / 3.0
    t = t.to(_DEV, _F64).reshape(-1, 1, 1)
    x = k * torch.arange(n, device=_DEV, dtype=_F64)
    sx, cx = torch.sin(x).reshape(1, 1, n), torch.cos(x).reshape(1, 1, n)
    sy, cy = torch.sin(x).reshape(1, n, 1), torch.cos(x).reshape(1, n, 1)
    a = -(amp * w / (2.0 * k)) * torch.sin(w * t)
    at = -(amp * w * w / (2.0 * k)) * torch.cos(w * t)
    p = _trig([(amp * torch.cos(w * t), "s", "s")], k, sx, cx, sy, cy)
    qx = _trig([(a, "c", "s"), (u0, "s", "c")], k, sx, cx, sy, cy)
    qy = _trig([(a, "s", "c"), (-u0, "c", "s")], k, sx, cx, sy, cy)
    p[""] = p[""] + phi0

    def over_phi(q):
        u = {"": q[""] / p[""]}
        for i in "xy":
            u[i] = (q[i] - u[""] * p[i]) / p[""]
        for i, j in ("xx", "xy", "yy"):
            u[i + j] = (q[i + j] - u[i] * p[j] - u[j] * p[i] - u[""] * p[i + j]) / p[""]
        return u

    u, v = over_phi(qx), over_phi(qy)
    div = u["x"] + v["y"]
    txx, tyy, txy = 2.0 * u["x"] - 2.0 / 3.0 * div, 2.0 * v["y"] - 2.0 / 3.0 * div, u["y"] + v["x"]
    dtx = u["xx"] + u["yy"] + (u["xx"] + v["xy"]) / 3.0
    dty = v["xx"] + v["yy"] + (u["xy"] + v["yy"]) / 3.0
    fx = at * cx * sy + qx["x"] * u[""] + qx[""] * u["x"] + qx["y"] * v[""] + qx[""] * v["y"]
    fy = at * sx * cy + qy["x"] * u[""] + qy[""] * u["x"] + qy["y"] * v[""] + qy[""] * v["y"]
    fx = fx - nu * (p["x"] * txx + p["y"] * txy + p[""] * dtx)
    fy = fy - nu * (p["x"] * txy + p["y"] * tyy + p[""] * dty)
    return p[""], u[""], v[""], torch.stack([fx, fy], dim=1)


_PERIOD = 1000


def _moving_inputs(c, seed):
    r = random.Random(int(seed))
    amp, u0 = r.uniform(0.15, 0.2), r.uniform(0.005, 0.01)
    phi, ux, uy, force = _manufactured(c["n"], torch.arange(_PERIOD), 0.8, amp, float(_PERIOD), u0)
    if c["storage"] != "fp64":
        phi, force = phi.float(), force.float()
    return phi, ux[0].contiguous(), uy[0].contiguous(), force


def _batch_lattices(c, seed):
    sizes = random.Random(c["mix"])
    r = random.Random(int(seed))
    out = []
    for _ in range(c["count"]):
        n = 32 + 16 * sizes.randint(0, 62)
        out.append(P.BatchLattice(n, r.uniform(0.55, 1.5), r.uniform(0.05, 0.3), 1000.0 * (n / 64.0) ** 2, 0.64 / n))
    return out


def _gradient_channel(c):
    return P.Channel(nx=c["nx"], ny=c["ny"], nsteps=c["nsteps"], avg_steps=c["avg"], checkpoint_every=c["every"])


# ---------------------------------------------------------------------- the cases
def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c, "kind": kind}
    if kind == "channel":
        phi, rho, u = _channel_inputs(c, seed)
        lat = P.Lattice(c["nx"], c["ny"], 0.6, s_e=1.2, s_eps=1.2, s_q=1.2, bc_y="bounceback", storage=c["storage"],
                        dev_base="momentum" if c.get("momentum") else "rest")
        if c.get("solid"):
            lat.set_solid_cells()
        lat.set_void_fraction(phi)
        lat.set_body_force(_gravity(c["ny"]), 0.0)
        if c.get("drag"):
            lat.set_drag(1e-3, 0.05)
        lat.init_fields(rho, u[0], u[1])
        s["lat"] = lat
    elif kind == "moving":
        phi, ux, uy, force = _moving_inputs(c, seed)
        lat = P.Lattice(c["n"], c["n"], 0.8, s_eps=1.2, s_q=1.2, storage=c["storage"])
        lat.set_void_fraction(phi[0])
        lat.set_body_force(0.0, 0.0, force[0])
        lat.init_fields(torch.ones_like(ux), ux, uy)
        s.update(lat=lat, phi=phi, force=force, t=0)
    elif kind == "cube":
        phi, rho, u = _cube_inputs(c, seed)
        lat = P.Lattice3D(c["nx"], c["ny"], c["nz"], 0.6, s_e=1.2, bc_y="bounceback", storage=c["storage"])
        lat.set_void_fraction(phi)
        lat.set_body_force(_gravity(c["ny"]), 0.0, 0.0)
        lat.init_fields(rho, u)
        s["lat"] = lat
    elif kind == "batch":
        b = P.Batch(_batch_lattices(c, seed), storage=c["storage"])
        b.init()
        s["batch"] = b
    else:
        s.update(phi=_porous((c["ny"], c["nx"]), _gen(seed)), channel=_gradient_channel(c))
    return s


def run(state):
    c, kind = state["case"], state["kind"]
    if kind == "gradient":
        value, grad, _ = P.outlet_momentum(state["phi"], state["channel"])
        return {"J": value, "grad": grad}
    keep = (lambda v: v) if c["storage"] == "fp64" else (lambda v: v.float())
    if kind == "batch":
        b = state["batch"]
        b.step(c["steps"])
        return [keep(b.populations(i)) for i in range(c["count"])]
    lat = state["lat"]
    if kind == "moving":
        phi, force = state["phi"], state["force"]
        for _ in range(c["steps"]):
            t = state["t"]
            state["t"] = (t + 1) % _PERIOD
            lat.set_void_fraction(phi[t], phi[state["t"]])
            lat.set_body_force(0.0, 0.0, force[t])
            lat.step(1)
    else:
        lat.step(c["steps"])
    out = {"f": keep(lat.get_populations())}
    if c.get("macros"):
        for name, v in lat.macros().items():
            out[name] = keep(v)
    return out


def work(case):
    """Bytes: the populations read and written and the fields read once a step, and the result
    written once. Flops of a cell's collision: about 300 (D2Q9) and 700 (D3Q19); a gradient
    steps forward and back, the way back costing about three collisions."""
    c, kind = case, case["kind"]
    if kind == "gradient":
        cells, n = c["nx"] * c["ny"], c["nsteps"]
        return {"bytes": float(cells * (n * (2 * 19 + 9) + 2) * 8), "flops": float(cells * n * 300 * 4)}
    z = _SIZE[c["storage"]]
    r, o = max(4, z), (8 if z == 8 else 4)
    if kind == "batch":
        sizes = random.Random(c["mix"])
        cells = sum((32 + 16 * sizes.randint(0, 62)) ** 2 for _ in range(c["count"]))
        return {"bytes": float(cells * (c["steps"] * 18 * z + 9 * o)), "flops": float(cells * c["steps"] * 400)}
    if kind == "cube":
        cells, q, fields, per = c["nx"] * c["ny"] * c["nz"], 19, 1, 700
    elif kind == "moving":
        cells, q, fields, per = c["n"] ** 2, 9, 4, 300
    else:
        cells, q, fields, per = c["nx"] * c["ny"], 9, 1, 300
    out = q + ((5 if q == 19 else 4) if c.get("macros") else 0)
    return {"bytes": float(cells * (c["steps"] * (2 * q * z + fields * r) + out * o)),
            "flops": float(cells * c["steps"] * per)}


# ---------------------------------------------------------------------- the scheme in 64 bits
# Arrays are [..., y, x] in 2-D and [z, y, x] in 3-D; axes from the right: x, y, z.
_E2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_E3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
       (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1)]


def _basis(e):
    """The moment polynomials at velocity e: nine in 2-D, nineteen in 3-D."""
    c2 = sum(v * v for v in e)
    if len(e) == 2:
        x, y = e
        return [1, 3 * c2 - 4, (9 * c2 * c2 - 21 * c2 + 8) // 2, x, (3 * c2 - 5) * x, y, (3 * c2 - 5) * y,
                x * x - y * y, x * y]
    x, y, z = e
    a, b = 3 * x * x - c2, y * y - z * z
    return [1, 19 * c2 - 30, (21 * c2 * c2 - 53 * c2 + 24) // 2, x, (5 * c2 - 9) * x, y, (5 * c2 - 9) * y, z,
            (5 * c2 - 9) * z, a, (3 * c2 - 5) * a, b, (3 * c2 - 5) * b, x * y, y * z, x * z, b * x,
            (z * z - x * x) * y, (x * x - y * y) * z]


class _Scheme:
    """One lattice of the scheme: e, w, M, the boundary rule and the rates."""

    def __init__(self, dim, rates, walls, kappa=0.5, solid=None, drag=(0.0, 0.0)):
        self.e = _E2 if dim == 2 else _E3
        self.dim, self.rates, self.walls, self.kappa, self.solid, self.drag = dim, rates, walls, kappa, solid, drag
        w = [4 / 9, 1 / 9, 1 / 36] if dim == 2 else [1 / 3, 1 / 18, 1 / 36]
        self.w = [w[sum(v * v for v in e)] for e in self.e]
        self.opp = [self.e.index(tuple(-v for v in e)) for e in self.e]
        self.M = [list(r) for r in zip(*[_basis(e) for e in self.e])]
        self.norm = [sum(v * v for v in r) for r in self.M]

    def at(self, v, e, odd=False):
        """v at x + e: x and z wrap, y wraps or mirrors about the wall (odd: sign changed)."""
        for ax, d in enumerate(e):
            if d and (ax != 1 or not self.walls):
                v = torch.roll(v, -d, -1 - ax)
        if e[1] and self.walls:
            edge = v[..., -1:, :] if e[1] > 0 else v[..., :1, :]
            edge = -edge if odd else edge
            v = torch.cat([v[..., 1:, :], edge] if e[1] > 0 else [edge, v[..., :-1, :]], -2)
        return v

    def neighbour(self, v, e, odd):
        a = self.at(v, e, odd)
        if self.solid is None:
            return a
        hit = self.at(self.solid, e)
        own = v
        if all(e):
            ax, ay = (e[0], 0), (0, e[1])
            fx, fy = ~self.at(self.solid, ax), ~self.at(self.solid, ay)
            gx, gy = self.at(v, ax, odd), self.at(v, ay, odd)
            own = torch.where(fx & fy, 0.5 * (gx + gy), torch.where(fx, gx, torch.where(fy, gy, v)))
        return torch.where(hit, -own if odd else own, a)

    def grad(self, v, odd, axes):
        out = [0.0] * self.dim
        for e, w in zip(self.e[1:], self.w[1:]):
            if any(e[a] for a in axes):
                n = self.neighbour(v, e, odd)
                for a in axes:
                    if e[a]:
                        out[a] = out[a] + 3.0 * w * e[a] * n
        return out

    def to_moments(self, f):
        return [sum(c * v for c, v in zip(row, f) if c) for row in self.M]

    def from_moments(self, m):
        m = [v / n for v, n in zip(m, self.norm)]
        return [sum(row[i] * v for row, v in zip(self.M, m) if row[i]) for i in range(len(self.e))]

    def force(self, rho, phi, fb):
        g = self.grad(rho, False, range(self.dim))
        return [(self.kappa - phi) / 3.0 * g[a] + fb[a] for a in range(self.dim)]

    def macros(self, f, phi, fb):
        m0 = sum(f)
        if self.solid is not None:
            m0 = torch.where(self.solid, torch.ones_like(m0), m0)
            phi = torch.where(self.solid, torch.ones_like(phi), phi)
        rho = m0 / phi
        F = self.force(rho, phi, fb)
        j = [sum(e[a] * v for e, v in zip(self.e, f) if e[a]) for a in range(self.dim)]
        beta = phi * phi * (self.drag[0] + self.drag[1] * (1.0 - phi))
        u = [(j[a] + 0.5 * F[a]) / (m0 + 0.5 * beta) for a in range(self.dim)]
        F = [F[a] - beta * u[a] for a in range(self.dim)]
        if self.solid is not None:
            u = [torch.where(self.solid, torch.zeros_like(v), v) for v in u]
        return m0, rho, phi, F, u

    def equilibrium(self, phi, rho, u):
        m0, X, k = phi * rho, self.kappa / phi, self.kappa
        uu = sum(v * v for v in u)
        z = torch.zeros_like(m0)
        if self.dim == 2:
            a = (X - 2.0) * m0
            return [m0, m0 * (-4.0 + 3.0 * uu + 2.0 * X), m0 * (4.0 - 3.0 * uu - 3.0 * X), m0 * u[0], a * u[0],
                    m0 * u[1], a * u[1], m0 * (u[0] * u[0] - u[1] * u[1]), m0 * u[0] * u[1]]
        q = (10.0 / 3.0 * X - 4.0) * m0
        a, b = m0 * (3.0 * u[0] * u[0] - uu), m0 * (u[1] * u[1] - u[2] * u[2])
        return [m0, 19.0 * (k * rho + m0 * uu) - 30.0 * m0, 12.0 * m0 - 9.0 * k * rho - 5.5 * m0 * uu, m0 * u[0],
                q * u[0], m0 * u[1], q * u[1], m0 * u[2], q * u[2], a, -0.5 * a, b, -0.5 * b, m0 * u[0] * u[1],
                m0 * u[1] * u[2], m0 * u[0] * u[2], z, z, z]

    def guo(self, u, F):
        out = []
        uF = sum(a * b for a, b in zip(u, F))
        for e, w in zip(self.e, self.w):
            eu = sum(a * b for a, b in zip(e, u) if a) if any(e) else 0.0
            eF = sum(a * b for a, b in zip(e, F) if a) if any(e) else 0.0
            out.append(w * (3.0 * (eF - uF) + 9.0 * eu * eF))
        return out

    def init(self, rho, u, phi, fb):
        if self.solid is not None:
            phi = torch.where(self.solid, torch.ones_like(phi), phi)
        F = self.force(rho, phi, fb)
        if any(self.drag):
            beta = phi * phi * (self.drag[0] + self.drag[1] * (1.0 - phi))
            F = [F[a] - beta * u[a] for a in range(self.dim)]
        f = [a - 0.5 * b for a, b in zip(self.from_moments(self.equilibrium(phi, rho, u)), self.guo(u, F))]
        return self.clear(f)

    def clear(self, f):
        if self.solid is None:
            return f
        return [torch.where(self.solid, torch.zeros_like(v), v) for v in f]

    def step(self, f, phi, phin, fb):
        m0, rho, phi, F, u = self.macros(f, phi, fb)
        k, X = self.kappa, self.kappa / phi
        kr = (k - phi) * rho
        n = self.dim
        B = [self.grad(u[a], True, range(n)) for a in range(n)]              # B[a][b] = d_b u_a
        A = [self.grad(rho * u[a], True, [a])[a] for a in range(n)]
        D = [self.grad(m0 * u[a], True, [a])[a] for a in range(n)]
        dphi = None if phin is None else phin - phi
        m, meq, S = self.to_moments(f), self.equilibrium(phi, rho, u), self.to_moments(self.guo(u, F))
        C = [0.0] * len(m)
        divB, divD = sum(B[a][a] for a in range(n)), sum(D)
        if n == 2:
            C[1] = -k * (A[0] + A[1]) + 2.0 * kr * divB + (3.0 - 2.0 * X) * divD
            if dphi is not None:
                C[1] = C[1] - 2.0 * X * rho * dphi
            C[7] = -k * (A[0] - A[1]) + 2.0 / 3.0 * kr * (B[0][0] - B[1][1]) + D[0] - D[1]
            C[8] = kr * (B[0][1] + B[1][0]) / 3.0
        else:
            C[1] = 19.0 * ((1.0 - X) * divD + 2.0 / 3.0 * kr * divB)
            d = [-k * A[a] + 2.0 / 3.0 * kr * B[a][a] + D[a] for a in range(3)]
            C[9], C[11] = 2.0 * d[0] - d[1] - d[2], d[1] - d[2]
            C[13], C[14], C[15] = (kr * (B[a][b] + B[b][a]) / 3.0 for a, b in ((0, 1), (1, 2), (0, 2)))
        m = [v - s * (v - q) + (1.0 - 0.5 * s) * (b + p) for v, q, b, p, s in zip(m, meq, S, C, self.rates)]
        fp = self.from_moments(m)
        out = []
        for i, e in enumerate(self.e):
            back = tuple(-v for v in e)
            v = fp[i]
            for ax, d in enumerate(e):
                if d:
                    v = torch.roll(v, d, -1 - ax)
            if self.walls and e[1]:
                o = fp[self.opp[i]]
                v = torch.cat([o[..., :1, :], v[..., 1:, :]] if e[1] > 0 else [v[..., :-1, :], o[..., -1:, :]], -2)
            if self.solid is not None and i:
                v = torch.where(self.at(self.solid, back), fp[self.opp[i]], v)
            out.append(v)
        return self.clear(out)


def _rates2(tau, s_e, s_eps=1.2, s_q=1.2):
    return [0.0, s_e, s_eps, 0.0, s_q, 0.0, s_q, 1.0 / tau, 1.0 / tau]


def _rates3(tau, s_e):
    n, s = 1.0 / tau, 1.2
    return [0.0, s_e, s, 0.0, s, 0.0, s, 0.0, s, n, s, n, s, n, n, n, s, s, s]


def _derived_s_e(tau):
    return 1.0 / ((tau - 0.5) / 3.0 + 0.5)


def _results(S, f, phi, fb, macros):
    out = {"f": torch.stack(f)}
    if macros:
        _, rho, _, _, u = S.macros(f, phi, fb)
        if S.solid is not None:
            rho = torch.where(S.solid, torch.zeros_like(rho), rho)
        out["rho"], out["p"] = rho, rho / 3.0
        out.update({"ux": u[0], "uy": u[1]} if S.dim == 2 else {"u": torch.stack(u)})
    return out


def _gradient(phi, c):
    """J and dJ/dphi by torch's reverse mode."""
    phi = phi.clone().requires_grad_(True)
    S = _Scheme(2, _rates2(0.6, 1.2), True)
    g = 1e-6
    fb = [g * phi, torch.zeros_like(phi)]
    one, zero = torch.ones_like(phi), torch.zeros_like(phi)
    f = S.init(one, [zero, zero], phi, fb)
    J = 0.0
    for n in range(c["nsteps"]):
        f = S.step(f, phi, None, fb)
        if n + 1 > c["nsteps"] - c["avg"]:
            m0, _, _, _, u = S.macros(f, phi, fb)
            J = J + (m0 * u[0])[:, -1].sum()
    J = J / (c["avg"] * c["ny"])
    return {"J": float(J.detach()), "grad": torch.autograd.grad(J, phi)[0]}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "gradient":
        return _gradient(_porous((c["ny"], c["nx"]), _gen(seed)), c)
    if kind == "channel":
        phi, rho, u = _channel_inputs(c, seed)
        S = _Scheme(2, _rates2(0.6, 1.2), True, solid=phi == 0 if c.get("solid") else None,
                    drag=(1e-3, 0.05) if c.get("drag") else (0.0, 0.0))
        fb = [_gravity(c["ny"]) * phi, torch.zeros_like(phi)]
        f = S.init(rho, u, phi, fb)
        for _ in range(c["steps"]):
            f = S.step(f, phi, None, fb)
        return _results(S, f, phi, fb, c.get("macros"))
    if kind == "cube":
        phi, rho, u = _cube_inputs(c, seed)
        S = _Scheme(3, _rates3(0.6, 1.2), True)
        fb = [_gravity(c["ny"]) * phi, torch.zeros_like(phi), torch.zeros_like(phi)]
        f = S.init(rho, list(u), phi, fb)
        for _ in range(c["steps"]):
            f = S.step(f, phi, None, fb)
        return _results(S, f, phi, fb, c.get("macros"))
    if kind == "moving":
        phi, ux, uy, force = (v.double() for v in _moving_inputs(c, seed))
        S = _Scheme(2, _rates2(0.8, _derived_s_e(0.8)), False)
        f = S.init(torch.ones_like(ux), [ux, uy], phi[0], force[0])
        for t in range(c["steps"]):
            f = S.step(f, phi[t], phi[t + 1], force[t])
        return _results(S, f, None, None, False)
    out = []
    for q in _batch_lattices(c, seed):
        t = torch.arange(c["steps"] + 1)
        S = _Scheme(2, _rates2(q.tau, 1.2), False)
        phi, ux, uy, force = _manufactured(q.n, t[:1], q.tau, q.amplitude, q.period, q.u0)
        f = S.init(torch.ones_like(phi[0]), [ux[0], uy[0]], phi[0], force[0])
        for k in range(c["steps"]):
            nxt, _, _, fnext = _manufactured(q.n, t[k + 1:k + 2], q.tau, q.amplitude, q.period, q.u0)
            f = S.step(f, phi[0], nxt[0], force[0])
            phi, force = nxt, fnext
        out.append(torch.stack(f))
    return out
