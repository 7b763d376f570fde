"""The work the performance of this framework is measured on.

Each case is one pass of a program that uses the package in earnest: steps of a channel with
held disks, coupled LBM-DEM cycles of a suspension or of a collapsing column, the drag gradient,
the batched sweep, and the D3Q19 lattice with held spheres.  `run` drives the public entry
points and returns what the pass computed; `exact` evaluates the same equations in 64 bits with
plain torch and numpy.

The C ABI hands every field and force out as FP64, widened from the type the populations are
stored in.  The outputs are given back in that storage type (forces and fields of an FP32
lattice as FP32, of a 16-bit lattice as 16 bits); particle positions, integrated in FP64, stay
FP64 with FP32 populations and are given as FP32 with 16-bit ones, whose forces move them.
"""
import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1809_07008_gb300 as imb

TYPES = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
F64 = torch.float64


def listed():
    return [
        # the 200 x 100 channel with one held disk (inlet, outlet, walls): the smallest lattice,
        # a step is two launches of a few microseconds
        dict(name="channel_200x100", kind="channel", nx=200, ny=100, disks=1, d=20.0, tau=0.6, C=0.0,
             u_in=0.02, storage="fp32", steps=100),
        # a host program that exchanges kinematics and forces every coupling cycle on a small
        # suspension: the smallest call, one cycle, all latency
        dict(name="loop_512x512", kind="suspension", nx=512, ny=512, phi=0.187, d=20.0, spread=0.0, gap=0.1,
             box=False, gravity=0.0, tau=0.51, C=0.1, storage="fp32", steps=1, fields=False),
        # the 8192 x 4096 suspension of 20 000 disks, the largest lattice, in FP32 and with
        # 16-bit populations
        dict(name="suspension_8192x4096_fp32", kind="suspension", nx=8192, ny=4096, phi=0.187, d=20.0, spread=0.0,
             gap=0.1, box=False, gravity=0.0, tau=0.51, C=0.1, storage="fp32", steps=60, fields=True),
        dict(name="suspension_8192x4096_fp16", kind="suspension", nx=8192, ny=4096, phi=0.187, d=20.0, spread=0.0,
             gap=0.1, box=False, gravity=0.0, tau=0.51, C=0.1, storage="fp16", steps=60, fields=True),
        # a dense suspension on a lattice of odd size, populations in bfloat16
        dict(name="suspension_1531x1087_bf16", kind="suspension", nx=1531, ny=1087, phi=0.40, d=20.0, spread=0.0,
             gap=0.1, box=False, gravity=0.0, tau=0.52, C=0.1, storage="bf16", steps=40, fields=True),
        # the settled column at the start of its collapse: 1000 disks of 16 to 24 cells stacked in
        # a closed box under gravity, in contact or about to be
        dict(name="collapse_2048x1024", kind="suspension", nx=2048, ny=1024, phi=0.15, d=20.0, spread=4.0, gap=0.02,
             box=True, gravity=1.0e-5, tau=0.52, C=0.1, storage="fp32", steps=10, fields=True),
        # the drag gradient of the 512 x 256 channel with 16 held disks: forward and reverse mode
        dict(name="gradient_512x256", kind="gradient", nx=512, ny=256, disks=16, d=20.0, tau=0.6, u_in=0.02,
             steps=400, every=50, snapshots=-1),
        # the parameter sweep: 256 periodic domains of 128 x 128 to 512 x 256 cells in FP16, and
        # a small one in FP32
        dict(name="sweep_256_fp16", kind="sweep", domains=256, lo=128, hi_x=512, hi_y=256, storage="fp16", steps=100),
        dict(name="sweep_12_fp32", kind="sweep", domains=12, lo=75, hi_x=260, hi_y=200, storage="fp32", steps=200),
        # D3Q19: Poiseuille flow past one sphere of 20 cells (the paper's first benchmark)
        dict(name="sphere_400x100x400_fp32", kind="spheres", nx=400, ny=100, nz=400, spheres=1, d=20.0, wall=True,
             tau=1.0, storage="fp32", steps=60),
        # D3Q19: several moving-surface spheres on an odd lattice with 16-bit populations
        dict(name="spheres_203x77x151_fp16", kind="spheres", nx=203, ny=77, nz=151, spheres=8, d=16.0, wall=True,
             tau=0.7, storage="fp16", steps=100),
        # D3Q19: the paper's packed bed, 250 touching spheres, Smagorinsky closure, half the
        # cells covered
        dict(name="packed_bed_240x100x100", kind="bed", N=20, tau=0.51, C=0.3, storage="fp32", steps=60),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel", "suspension", "suspension", "suspension", "gradient", "sweep", "spheres", "bed"])
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    if kind == "channel":
        nx, ny = _log(rng, 180, 3000), _log(rng, 90, 1500)
        return dict(kind=kind, nx=nx, ny=ny, disks=rng.choice([1, 1, 4, 9]), d=round(rng.uniform(8.0, 21.0), 2),
                    tau=round(rng.uniform(0.55, 0.9), 3), C=rng.choice([0.0, 0.1]), u_in=0.02, storage=storage,
                    steps=rng.randint(60, 120))
    if kind == "suspension":
        nx, ny = _log(rng, 300, 8192), _log(rng, 300, 4096)
        small = nx * ny < 400_000
        return dict(kind=kind, nx=nx, ny=ny, phi=round(rng.uniform(0.05, 0.42), 3), d=round(rng.uniform(12.0, 24.0), 2),
                    spread=0.0, gap=0.1, box=False, gravity=0.0, tau=round(rng.uniform(0.51, 0.6), 3), C=0.1,
                    storage=storage, steps=1 if small else rng.randint(20, 50), fields=not small)
    if kind == "gradient":
        return dict(kind=kind, nx=_log(rng, 300, 1200), ny=_log(rng, 200, 600), disks=rng.choice([4, 9, 16]),
                    d=round(rng.uniform(12.0, 22.0), 2), tau=round(rng.uniform(0.55, 0.8), 3), u_in=0.02,
                    steps=rng.randint(60, 240), every=rng.choice([20, 50]), snapshots=rng.choice([-1, 5]))
    if kind == "sweep":
        return dict(kind=kind, domains=_log(rng, 6, 200), lo=rng.randint(70, 128), hi_x=rng.randint(200, 512),
                    hi_y=rng.randint(150, 256), storage=storage, steps=rng.randint(60, 120))
    if kind == "spheres":
        return dict(kind=kind, nx=_log(rng, 60, 420), ny=_log(rng, 40, 110), nz=_log(rng, 60, 400),
                    spheres=rng.choice([1, 3, 6]), d=round(rng.uniform(8.0, 16.0), 2), wall=rng.random() < 0.7,
                    tau=round(rng.uniform(0.55, 1.0), 3), storage=storage, steps=rng.randint(30, 60))
    return dict(kind="bed", N=rng.choice([8, 11, 14, 17]), tau=round(rng.uniform(0.51, 0.58), 3),
                C=rng.choice([0.1, 0.3]), storage=storage, steps=rng.randint(30, 60))


# ------------------------------------------------------------------------------ inputs
def _grid(g, nx, ny, n, d, gap):
    """n disks on a jittered grid, at least `gap` apart and gap / 2 from the edges."""
    cols = max(1, min(int(math.sqrt(n * nx / ny)), int(nx // (d + gap))))
    rows = min(-(-n // cols), int(ny // (d + gap)))
    sx, sy = nx / cols, ny / rows
    site = g.permutation(cols * rows)[: min(n, cols * rows)]
    site.sort()
    jx, jy = (sx - d - gap) / 2, (sy - d - gap) / 2
    x = (site % cols + 0.5) * sx + g.uniform(-jx, jx, site.size)
    y = (site // cols + 0.5) * sy + g.uniform(-jy, jy, site.size)
    return np.stack([x, y], 1)


def _stack(g, nx, ny, n, d, spread, gap):
    """Columns of disks of diameter d -+ spread resting on one another, up to `gap` apart."""
    pitch = d + spread + gap
    cols = max(1, min(int(0.32 * nx / pitch), n))
    dia = g.uniform(d - spread, d + spread, n)
    gaps = g.uniform(0.1 * gap, gap, n)
    x, y, r, top = [], [], [], np.zeros(cols)
    for k in range(n):
        c = k % cols
        y0 = top[c] + gaps[k] + dia[k] / 2
        if y0 + dia[k] / 2 + 1.0 > ny:
            continue
        top[c] = y0 + dia[k] / 2
        x.append((c + 0.5) * pitch + gap)
        y.append(y0)
        r.append(dia[k] / 2)
    return np.stack([x, y], 1), np.array(r)


def _disks(case, seed):
    """Centres, velocities, spins and radii of the disks of a 2D case."""
    g = np.random.default_rng(seed)
    nx, ny, d = case["nx"], case["ny"], case["d"]
    if case["kind"] != "suspension":
        side = max(1, int(math.isqrt(case["disks"])))
        sx, sy = nx / (side + 1), ny / (side + 1)
        i = np.arange(side * side)
        x = np.stack([(i % side + 1) * sx, (i // side + 1) * sy], 1) + 0.1 * min(sx, sy) * g.uniform(-1, 1, (side * side, 2))
        d = min(d, 0.7 * min(sx, sy))
        n = len(x)
        return x, np.zeros((n, 2)), np.zeros(n), np.full(n, d / 2)
    n = max(1, int(round(case["phi"] * nx * ny / (math.pi * d * d / 4))))
    if case["box"]:
        x, r = _stack(g, nx, ny, n, d, case["spread"], case["gap"])
    else:
        x = _grid(g, nx, ny, n, d, case["gap"])
        r = np.full(len(x), d / 2)
    a = g.uniform(0, 2 * math.pi, len(x))
    v = 0.005 * np.stack([np.cos(a), np.sin(a)], 1)
    return x, v, g.uniform(-1e-4, 1e-4, len(x)), r


def _domains(case, seed):
    g = np.random.default_rng(seed)
    out = []
    for _ in range(case["domains"]):
        nx, ny = int(g.integers(case["lo"], case["hi_x"] + 1)), int(g.integers(case["lo"], case["hi_y"] + 1))
        d, phi, tau = g.uniform(10.0, 30.0), g.uniform(0.1, 0.5), g.uniform(0.51, 1.0)
        Re, nu = 10.0 ** g.uniform(-1.0, 2.0), 0.0
        n = max(1, int(round(phi * nx * ny / (math.pi * d * d / 4))))
        x = _grid(g, nx, ny, n, d, 0.5)
        phi, nu = len(x) * math.pi * d * d / 4 / (nx * ny), (tau - 0.5) / 3
        force = nu * min(Re * nu / d, 0.02) / (d * d * (1 - phi) ** 3 / (9 * phi * phi))
        out.append(SimpleNamespace(nx=nx, ny=ny, tau=tau, C_smag=0.1, force=(force, 0.0), n_particles=len(x), x=x,
                                   r=np.full(len(x), d / 2)))
    return out


def _spheres(case, seed):
    g = np.random.default_rng(seed)
    if case["kind"] == "bed":
        N, tau = case["N"], case["tau"]
        off = g.uniform(0.35, 0.65, 3)
        i, j, k = np.meshgrid(np.arange(10), np.arange(5), np.arange(5), indexing="ij")
        x = np.stack([(1.5 + i) * N, (0.5 + j) * N, (0.5 + k) * N], -1).reshape(-1, 3) + off
        # the paper's pressure differences go as 1 / (tau - 1/2)^2, 50 Pa at tau = 0.51
        force = (50.0 / 0.01) * (0.01 / 3 * (1e-3 / N) ** 2 / 1e-6) ** 2 / (1000.0 * 1e-3 / N) * g.uniform(0.8, 1.2)
        return SimpleNamespace(nx=12 * N, ny=5 * N, nz=5 * N, tau=tau, C=case["C"], wall=False, force=(force, 0.0, 0.0), x=x,
                               v=np.zeros_like(x), w=np.zeros_like(x), R=np.full(len(x), N / 2))
    L, d, x = np.array([case["nx"], case["ny"], case["nz"]], float), min(case["d"], 0.4 * case["ny"]), []
    one = case["spheres"] == 1
    for _ in range(400):
        c = L * (0.5, 0.25, 0.5) + g.uniform(-0.5, 0.5, 3) if one else g.uniform(0, 1, 3) * L
        if len(x) == case["spheres"] or (case["wall"] and not d / 2 + 1 < c[1] < L[1] - d / 2 - 1):
            continue
        e = np.array(x).reshape(-1, 3) - c
        e -= L * np.round(e / L)
        if not len(x) or (e * e).sum(1).min() > (d + 2) ** 2:
            x.append(c)
    x = np.array(x).reshape(-1, 3)
    H, nu = L[1], (case["tau"] - 0.5) / 3
    v = np.zeros_like(x) if one else g.uniform(-2e-3, 2e-3, x.shape)
    return SimpleNamespace(nx=case["nx"], ny=case["ny"], nz=case["nz"], tau=case["tau"], C=0.0, wall=case["wall"],
                           force=(2e-4 * 32 * nu / (3 * H * H) * g.uniform(0.8, 1.2), 0.0, 0.0), x=x, v=v, w=0.1 * v,
                           R=np.full(len(x), d / 2))


# ------------------------------------------------------------------------ prepare and run
def _pinned(*shape):
    return torch.zeros(shape, dtype=F64, pin_memory=True)


def _ptr(t):
    return ctypes.cast(t.data_ptr(), ctypes.POINTER(ctypes.c_double))


def prepare(case, seed):
    s = SimpleNamespace(case=case, kind=case["kind"], n=case["steps"], type=TYPES[case.get("storage", "fp32")])
    if s.kind == "sweep":
        s.lat = imb.Batch(_domains(case, seed), storage=case["storage"])
        s.lat.autotune(5)   # as a sweep does once before its thousands of steps
        return s
    if s.kind in ("spheres", "bed"):
        p = _spheres(case, seed)
        s.lat = imb.Lattice3(p.nx, p.ny, p.nz, p.tau, wall_y=p.wall, force=p.force, storage=case["storage"], C_smag=p.C)
        s.lat.set_spheres(p.x, p.v, p.w, p.R)
        s.fields = _pinned(4, p.nz, p.ny, p.nx)
        return s
    x, v, w, r = _disks(case, seed)
    kw = dict(storage=case.get("storage", "fp32"))
    if s.kind == "suspension":
        kw |= dict(bc_x=imb.BC_WALL if case["box"] else imb.BC_PERIODIC, bc_y=imb.BC_WALL, dem_on=1, gy=-case["gravity"])
    else:
        kw |= dict(bc_x=imb.BC_INLET_OUTLET, bc_y=imb.BC_WALL, u_in_x=case["u_in"], ux0=case["u_in"])
    s.lat = imb.Lattice(case["nx"], case["ny"], case["tau"], case.get("C", 0.0), **kw)
    s.lat.set_particles(x, v, w, r)
    if s.kind == "suspension":
        n = len(r)
        s.kin, s.io = [_pinned(n, 2), _pinned(n, 2), _pinned(n)], [_pinned(n, 2), _pinned(n), _pinned(n, 2), _pinned(n, 2), _pinned(n)]
        for t, a in zip(s.kin, (x, v, w)):
            t.copy_(torch.from_numpy(a))
        s.kin_np, s.io_np = [t.numpy() for t in s.kin], [t.numpy() for t in s.io]
    if s.kind == "channel" or case.get("fields"):
        s.fields = _pinned(3, case["ny"], case["nx"])
    return s


def _macro(s):
    """The macroscopic fields, read back into pinned memory and handed on to the GPU program."""
    f, lib = s.fields, imb.load()
    rc = (lib.imb_get_macro if f.shape[0] == 3 else lib.imb3_get_macro)(s.lat.h, *(_ptr(f[k]) for k in range(f.shape[0])))
    if rc:
        raise imb.ImbError(rc, "macroscopic fields")
    g = f.to("cuda")
    return [g[k].to(s.type) for k in range(f.shape[0])]


def run(s):
    t = lambda a: torch.as_tensor(a).to(s.type)  # noqa: E731
    if s.kind == "suspension":
        # the host owns the kinematics at the start of the pass, the coupled cycles move them on
        F, T, x, v, w = s.io_np
        s.lat.step_io(s.n, kin_in=s.kin_np, F=F, T=T, x=x, v=v, w=w)
        out = dict(loads=t(np.column_stack([F, T])), x=s.io[2] if s.type == torch.float32 else s.io[2].float(), v=t(v), w=t(w))
        if s.case["fields"]:
            out["fields"] = _macro(s)
        return out
    if s.kind == "gradient":
        k = s.case["snapshots"]
        J, du, dtau, dx = s.lat.drag_gradient(s.n, s.case["every"], None if k < 0 else k)
        return dict(J=t(J), duin=t(du), dtau=t(dtau), dx=t(dx))
    if s.kind == "sweep":
        s.lat.run(s.n)
        return dict(drag=t(np.stack(s.lat.mean_drag(), 1)))
    s.lat.step(s.n)
    F, T = s.lat.forces()
    return dict(loads=t(np.column_stack([F, T])), fields=_macro(s))


def work(case):
    size = 4 if case.get("storage", "fp32") == "fp32" else 2
    if case["kind"] == "sweep":   # mean domain size; the solid ratio is read with every step
        cells = case["domains"] * (case["lo"] + case["hi_x"]) / 2 * (case["lo"] + case["hi_y"]) / 2
        return dict(bytes=case["steps"] * cells * (18 * size + 4), flops=case["steps"] * cells * 250.0)
    if case["kind"] == "bed":
        cells = 300.0 * case["N"] ** 3
        return dict(bytes=case["steps"] * cells * (38 * size + 4) + 32 * cells, flops=case["steps"] * cells * 700.0)
    if case["kind"] == "spheres":
        cells = float(case["nx"] * case["ny"] * case["nz"])
        return dict(bytes=case["steps"] * cells * (38 * size + 4) + 32 * cells, flops=case["steps"] * cells * 500.0)
    cells = float(case["nx"] * case["ny"])
    if case["kind"] == "gradient":   # a forward and a reverse step each: 72 and 112 bytes a cell
        return dict(bytes=case["steps"] * cells * 184, flops=case["steps"] * cells * 700.0)
    out = 24 * cells if case["kind"] == "channel" or case["fields"] else 0
    n = case["phi"] * cells / (math.pi * case["d"] ** 2 / 4) if case["kind"] == "suspension" else 0
    return dict(bytes=case["steps"] * cells * 18 * size + out, flops=case["steps"] * (cells * 250.0 + n * 1000))


# -------------------------------------------------------------------- the same in 64 bits
DEV = "cuda" if torch.cuda.is_available() else "cpu"
C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
      (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


def _weight(c):
    k = sum(abs(a) for a in c)
    return ((4 / 9, 1 / 9, 1 / 36) if len(c) == 2 else (1 / 3, 1 / 18, 1 / 36))[k]


def _dot(c, v):
    return sum((k * a for k, a in zip(c, v) if k), start=0.0)


class _Model:
    """D2Q9 or D3Q19, planes [.., y, x]: pull streaming with the boundary rules (Eq. 1), BGK with
    Smagorinsky relaxation time and Guo forcing, immersed moving boundary (Eqs. 12-16)."""

    def __init__(self, size, tau, C, force, bc_x="periodic", bc_y="periodic", u_in=0.0):
        self.C = C2 if len(size) == 2 else C3
        self.W = [_weight(c) for c in self.C]
        self.opp = [self.C.index(tuple(-a for a in c)) for c in self.C]
        self.shape, self.tau, self.Cs, self.F = tuple(reversed(size)), tau, C, force
        self.bc_x, self.bc_y, self.u_in = bc_x, bc_y, u_in

    def start(self):
        """The uniform equilibrium the lattices begin with, at the inlet's velocity."""
        u = [torch.full(self.shape, self.u_in if k == 0 else 0.0, dtype=F64, device=DEV) for k in range(len(self.C[0]))]
        return list(self.equilibrium(1.0, u))

    def equilibrium(self, rho, u):
        uu = sum(a * a for a in u)
        for c, w in zip(self.C, self.W):
            cu = _dot(c, u)
            yield w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)

    def pull(self, f):
        g = []
        for q, c in enumerate(self.C):
            h = torch.roll(f[q], tuple(reversed(c)), tuple(range(len(c)))) if any(c) else f[q].clone()
            back = f[self.opp[q]]
            if self.bc_x == "wall" and c[0]:
                i = 0 if c[0] > 0 else -1
                h[..., i] = back[..., i]
            if self.bc_y == "wall" and c[1]:
                i = 0 if c[1] > 0 else -1
                h[..., i, :] = back[..., i, :]
            g.append(h)
        if self.bc_x == "inlet":
            rho1 = sum(h[:, 1] for h in g)
            rho2 = sum(h[:, -2] for h in g)
            u2 = [sum(c[k] * h[:, -2] for c, h in zip(self.C, g)) / rho2 for k in (0, 1)]
            first = list(self.equilibrium(rho1, (self.u_in + 0 * rho1, 0 * rho1)))
            last = list(self.equilibrium(1 + 0 * rho2, u2))
            g = [torch.cat([a[:, None], h[:, 1:-1], b[:, None]], 1) for a, h, b in zip(first, g, last)]
        return g

    def moments(self, f):
        rho = sum(f[1:], start=f[0].clone())
        j = [_dot_planes(self.C, f, k) + 0.5 * self.F[k] for k in range(len(self.C[0]))]
        return rho, j

    def collide(self, f, E, solid=None, tau=None):
        """f, the summed solid ratio E of each cell (None: no solid) and the eps-weighted sums of
        the surface velocities (u, u u) over the bodies on a cell -> post-collision f, B, rho, j."""
        tau = self.tau if tau is None else tau
        rho, j = self.moments(f)
        u = [a / rho for a in j]
        n = [a - b for a, b in zip(f, self.equilibrium(rho, u))]
        te = tau
        if not (isinstance(self.Cs, float) and self.Cs == 0.0):
            D, Q = len(u), 0.0
            for a in range(D):
                for b in range(a, D):
                    P = sum(c[a] * c[b] * m for c, m in zip(self.C, n) if c[a] * c[b])
                    Q = Q + (1 if a == b else 2) * P * P
            te = 0.5 * (tau + torch.sqrt(tau * tau + 18 * math.sqrt(2) * self.Cs ** 2 * torch.sqrt(Q) / rho))
        B = 0.0
        if E is not None:
            e, tm = E.clamp(max=1.0), te - 0.5
            B = e * tm / ((1 - e) + tm)
        uF, out = sum(a * b for a, b in zip(u, self.F)), []
        share = B / E.clamp(min=1e-300) if solid is not None else None
        for q, (c, w) in enumerate(zip(self.C, self.W)):
            fluid = -n[q] / te
            if any(isinstance(a, torch.Tensor) or a for a in self.F):
                cF = _dot(c, self.F)
                fluid = fluid + (1 - 0.5 / te) * w * (3 * (cF - uF) + 9 * _dot(c, u) * cF)
            g = f[q] + (1 - B) * fluid
            if E is not None:   # sum_p B_p (f_-q - feq_-q(u) + feq_q(u_s) - f_q)
                eq = B
                if solid is not None:
                    s1, s2 = solid
                    cc = sum((1 if a == b else 2) * c[a] * c[b] * m for (a, b), m in s2.items() if c[a] * c[b])
                    tr = sum(m for (a, b), m in s2.items() if a == b)
                    eq = eq + share * (3 * _dot(c, s1) + 4.5 * cc - 1.5 * tr)
                g = g + B * (n[self.opp[q]] - f[q]) + w * rho * eq
            out.append(g)
        return out, B, rho, j


def _dot_planes(C, f, k):
    return sum((f[q] if c[k] > 0 else -f[q]) for q, c in enumerate(C) if c[k])


def _disk_cells(x, r, size, per):
    """(body, flat cell, overlap area, node minus centre) of every cell the disks reach into."""
    nx, ny = size
    X, R = torch.as_tensor(x, dtype=F64, device=DEV), torch.as_tensor(r, dtype=F64, device=DEV)
    h = int(math.ceil(float(R.max()))) + 1
    o = torch.arange(-h, h + 1, device=DEV)
    c = torch.floor(X)
    lo = [(o[None, :].to(F64) - (X - c)[:, k:k + 1]) for k in (0, 1)]
    x0, y0, rr = lo[0][:, None, :], lo[1][:, :, None], R[:, None, None]
    i, k = c[:, 0, None, None].long() + o[None, None, :], c[:, 1, None, None].long() + o[None, :, None]
    i, k, x0, y0, rr = torch.broadcast_tensors(i, k, x0, y0, rr)
    far = torch.maximum(x0.abs(), (x0 + 1).abs()) ** 2 + torch.maximum(y0.abs(), (y0 + 1).abs()) ** 2
    near = x0.clamp(min=0) ** 2 + (-(x0 + 1)).clamp(min=0) ** 2 + y0.clamp(min=0) ** 2 + (-(y0 + 1)).clamp(min=0) ** 2
    keep = near < rr * rr
    for a, L, p in ((i, nx, per[0]), (k, ny, per[1])):
        if not p:
            keep = keep & (a >= 0) & (a < L)
    body = torch.arange(len(X), device=DEV)[:, None, None].expand_as(keep)[keep]
    i, k, x0, y0, rr, far = (a[keep] for a in (i, k, x0, y0, rr, far))
    area = torch.ones_like(x0)
    part = far > rr * rr
    area[part] = _overlap(x0[part], y0[part], rr[part])
    return body, (k % ny) * nx + i % nx, area, (x0 + 0.5, y0 + 0.5)


def _overlap(x0, y0, r):
    """Area of the disk of radius r about the origin in [x0, x0 + 1] x [y0, y0 + 1]: with
    h = sqrt(r^2 - x^2) and M(y) the integral of max(h - y, 0) over the cell's columns,
    M(y0) - M(y1) + M(-y1) - M(-y0) - (columns)."""
    a, b = torch.maximum(x0, -r), torch.minimum(x0 + 1, r)

    def M(y):
        s = torch.where(y > 0, torch.sqrt((r * r - y * y).clamp(min=0)), r)
        p, q = torch.maximum(a, -s), torch.minimum(b, s)
        q = torch.maximum(p, q)

        def H(t):
            return 0.5 * (t * torch.sqrt((r * r - t * t).clamp(min=0)) + r * r * torch.asin((t / r).clamp(-1, 1)))
        return H(q) - H(p) - y * (q - p)
    return (M(y0) - M(y0 + 1) - (b - a).clamp(min=0) - M(-y0) + M(-y0 - 1)).clamp(0, 1)


def _solid_sums(shape, body, cell, eps, us):
    """Summed solid ratio and the eps-weighted sums of u_s and u_s u_s per cell."""
    def add(v):
        return torch.zeros(math.prod(shape), dtype=F64, device=DEV).index_add_(0, cell, v).view(shape)
    D = len(us)
    return add(eps), ([add(eps * a) for a in us], {(a, b): add(eps * us[a] * us[b]) for a in range(D) for b in range(a, D)})


def _body_sum(n, body, v):
    return torch.zeros(n, dtype=F64, device=DEV).index_add_(0, body, v)


class _Dem:
    """Disks with linear spring-dashpot contacts between them and with the walls (Eqs. 7-11), 100
    leapfrog sub-cycles a lattice step."""

    def __init__(self, x, v, w, r, size, per, gravity):
        self.x, self.v, self.w, self.r = (torch.as_tensor(a, dtype=F64, device=DEV).clone() for a in (x, v, w, r))
        self.m = 2.65 * math.pi * self.r ** 2
        self.I = 0.5 * self.m * self.r ** 2
        self.size, self.per = size, per
        self.g = -gravity * (1 - 1 / 2.65)
        self.wall = torch.zeros((4, len(r)), dtype=F64, device=DEV)
        self.pairs, self.xi = torch.zeros((0, 2), dtype=torch.long, device=DEV), torch.zeros(0, dtype=F64, device=DEV)

    def image(self, d):
        for k in (0, 1):
            if self.per[k]:
                d[..., k] -= self.size[k] * torch.round(d[..., k] / self.size[k])
        return d

    def neighbours(self):
        n, found = len(self.r), []
        for lo in range(0, n, 2000):
            d = self.image(self.x[None, :, :] - self.x[lo:lo + 2000, None, :])
            R = self.r[None, :] + self.r[lo:lo + 2000, None] + 1.0
            hit = ((d * d).sum(-1) < R * R).nonzero()
            hit[:, 0] += lo
            found.append(hit[hit[:, 0] < hit[:, 1]])
        new = torch.cat(found)
        key, old = new[:, 0] * n + new[:, 1], self.pairs[:, 0] * n + self.pairs[:, 1]
        xi = torch.zeros(len(new), dtype=F64, device=DEV)
        if len(old):
            at = torch.searchsorted(old, key).clamp(max=len(old) - 1)
            xi = torch.where(old[at] == key, self.xi[at], xi)
        self.pairs, self.xi = new, xi

    def law(self, nx, ny, delta, dvx, dvy, rot, cn, xi, dt):
        kn, kt, ct = 1e5, 0.5e5, 0.5 * cn
        tx, ty = -ny, nx
        vt = dvx * tx + dvy * ty - rot
        xi = xi + vt * dt
        Fn = kn * delta - cn * (dvx * nx + dvy * ny)
        Ft, lim = kt * xi + ct * vt, 0.5 * Fn.abs()
        slip = Ft.abs() > lim
        Ft, xi = torch.where(slip, torch.copysign(lim, Ft), Ft), torch.where(slip, torch.copysign(lim / kt, xi), xi)
        return -Fn * nx + Ft * tx, -Fn * ny + Ft * ty, Ft, xi

    def cycle(self, F, T):
        self.neighbours()
        dt, le = 0.01, math.log(0.5)
        zeta = -le / math.sqrt(math.pi ** 2 + le * le)
        a, b = self.pairs[:, 0], self.pairs[:, 1]
        ms = self.m[a] * self.m[b] / (self.m[a] + self.m[b])
        cn, cw = 2 * zeta * torch.sqrt(ms * 1e5), 2 * zeta * torch.sqrt(self.m * 1e5)
        R = self.r[a] + self.r[b]
        for _ in range(100):
            f, tq = F.clone(), T.clone()
            if len(a):
                d = self.image(self.x[b] - self.x[a])
                dist = torch.sqrt((d * d).sum(-1))
                on = dist < R
                n = d / dist[:, None]
                dv = self.v[b] - self.v[a]
                fx, fy, Ft, xi = self.law(n[:, 0], n[:, 1], R - dist, dv[:, 0], dv[:, 1],
                                          self.w[a] * self.r[a] + self.w[b] * self.r[b], cn, self.xi, dt)
                self.xi = torch.where(on, xi, 0.0 * xi)
                p, Ft = torch.stack([fx, fy], 1) * on[:, None], Ft * on
                f.index_add_(0, a, p).index_add_(0, b, -p)
                tq.index_add_(0, a, self.r[a] * Ft).index_add_(0, b, self.r[b] * Ft)
            for k, (ax, side) in enumerate(((0, 0), (0, 1), (1, 0), (1, 1))):
                if self.per[ax]:
                    continue
                dist = self.size[ax] - self.x[:, ax] if side else self.x[:, ax]
                on, s = dist < self.r, 1.0 if side else -1.0
                nx, ny = (s, 0.0) if ax == 0 else (0.0, s)
                fx, fy, Ft, xi = self.law(nx, ny, self.r - dist, -self.v[:, 0], -self.v[:, 1], self.w * self.r, cw, self.wall[k], dt)
                self.wall[k] = torch.where(on, xi, 0.0 * xi)
                f += torch.stack([fx, fy], 1) * on[:, None]
                tq += self.r * Ft * on
            self.v = self.v + (f / self.m[:, None] + torch.tensor([0.0, self.g], dtype=F64, device=DEV)) * dt
            self.w = self.w + tq / self.I * dt
            self.x = self.x + self.v * dt
            for k in (0, 1):
                if self.per[k]:
                    self.x[:, k] = self.x[:, k] % self.size[k]


def _fields(M, f):
    rho, j = M.moments(M.pull(f))
    return [rho] + [a / rho for a in j]


def _exact_2d(case, seed):
    x, v, w, r = _disks(case, seed)
    size, n, coupled = (case["nx"], case["ny"]), len(r), case["kind"] == "suspension"
    per = (coupled and not case["box"], False)
    M = _Model(size, case["tau"], case["C"], (0.0, 0.0), "inlet" if not coupled else "periodic" if per[0] else "wall", "wall",
               case.get("u_in", 0.0))
    dem = _Dem(x, v, w, r, size, per, case.get("gravity", 0.0))
    f, F, T, cells = M.start(), torch.zeros((n, 2), dtype=F64, device=DEV), torch.zeros(n, dtype=F64, device=DEV), None
    for _ in range(case["steps"]):
        if coupled:
            dem.cycle(F, T)
        if coupled or cells is None:
            cells = _disk_cells(dem.x, dem.r, size, per)
            body, cell, eps, arm = cells
            us = [dem.v[body, 0] - dem.w[body] * arm[1], dem.v[body, 1] + dem.w[body] * arm[0]]
            E, solid = _solid_sums(M.shape, body, cell, eps, us)
        f, B, rho, j = M.collide(M.pull(f), E, solid)
        Bp = (B.view(-1)[cell] / E.view(-1)[cell].clamp(min=1e-300)) * eps
        k = [Bp * (j[a].view(-1)[cell] - rho.view(-1)[cell] * us[a]) for a in (0, 1)]
        F = torch.stack([_body_sum(n, body, a) for a in k], 1)
        T = _body_sum(n, body, arm[0] * k[1] - arm[1] * k[0])
    out = dict(loads=torch.cat([F, T[:, None]], 1))
    if coupled:
        out |= dict(x=dem.x, v=dem.v, w=dem.w)
    if not coupled or case["fields"]:
        out["fields"] = _fields(M, f)
    return out


def _exact_3d(case, seed):
    p = _spheres(case, seed)
    size, n, ns = (p.nx, p.ny, p.nz), len(p.R), 5
    M = _Model(size, p.tau, p.C, p.force, "periodic", "wall" if p.wall else "periodic")
    sub = (torch.arange(ns, dtype=F64, device=DEV) + 0.5) / ns
    found = []
    for s in range(n):   # the solid ratio: sub-cell centres inside the sphere
        h = int(math.ceil(p.R[s])) + 1
        o, c = torch.arange(-h, h + 1, dtype=F64, device=DEV), np.floor(p.x[s])
        q = [(((o[:, None] + sub[None, :]) - (p.x[s][k] - c[k])).reshape(-1)) ** 2 for k in range(3)]
        W = 2 * h + 1
        inside = (q[2][:, None, None] + (q[1][None, :, None] + q[0][None, None, :])) <= p.R[s] ** 2
        cnt = inside.view(W, ns, W, ns, W, ns).sum((1, 3, 5))
        at = cnt.nonzero()
        ijk = [at[:, 2 - k] - h + int(c[k]) for k in range(3)]
        keep = (ijk[1] >= 0) & (ijk[1] < p.ny) if p.wall else torch.ones_like(ijk[1], dtype=torch.bool)
        arm = [ijk[k].to(F64) + 0.5 - p.x[s][k] for k in range(3)]
        cell = ((ijk[2] % p.nz) * p.ny + ijk[1] % p.ny) * p.nx + ijk[0] % p.nx
        found.append([a[keep] for a in (torch.full_like(cell, s), cell, cnt[cnt > 0].to(F64) / ns ** 3, *arm)])
    body, cell, eps, *arm = (torch.cat(a) for a in zip(*found))
    v, w = (torch.as_tensor(a, dtype=F64, device=DEV)[body] for a in (p.v, p.w))
    us = [v[:, k] + w[:, (k + 1) % 3] * arm[(k + 2) % 3] - w[:, (k + 2) % 3] * arm[(k + 1) % 3] for k in range(3)]
    E, solid = _solid_sums(M.shape, body, cell, eps, us)
    f = M.start()
    for _ in range(case["steps"]):
        f, B, rho, j = M.collide(M.pull(f), E, solid)
    Bp = (B.view(-1)[cell] / E.view(-1)[cell].clamp(min=1e-300)) * eps
    k = [Bp * (j[a].view(-1)[cell] - rho.view(-1)[cell] * us[a] - p.force[a]) for a in range(3)]
    F = torch.stack([_body_sum(n, body, a) for a in k], 1)
    T = torch.stack([_body_sum(n, body, arm[(a + 1) % 3] * k[(a + 2) % 3] - arm[(a + 2) % 3] * k[(a + 1) % 3]) for a in range(3)], 1)
    return dict(loads=torch.cat([F, T], 1), fields=_fields(M, f))


def _exact_sweep(case, seed):
    """All domains as one row of cells, streamed by gathering from each cell's periodic neighbour."""
    doms, start, src, E, par = _domains(case, seed), 0, [[] for _ in C2], [], []
    for d in doms:
        n = torch.arange(d.nx * d.ny, device=DEV)
        i, k = n % d.nx, n // d.nx
        for q, c in enumerate(C2):
            src[q].append(start + ((k - c[1]) % d.ny) * d.nx + (i - c[0]) % d.nx)
        body, cell, eps, _ = _disk_cells(d.x, d.r, (d.nx, d.ny), (True, True))
        E.append(torch.zeros(d.nx * d.ny, dtype=F64, device=DEV).index_add_(0, cell, eps))
        start += d.nx * d.ny
    num = torch.tensor([d.nx * d.ny for d in doms], device=DEV)
    dom = torch.repeat_interleave(torch.arange(len(doms), device=DEV), num)
    tau, Fx = (torch.tensor(a, dtype=F64, device=DEV)[dom] for a in ([d.tau for d in doms], [d.force[0] for d in doms]))
    src, E = [torch.cat(a) for a in src], torch.cat(E)
    M = _Model((start, 1), tau, 0.1, (Fx, 0.0))
    M.shape = (start,)
    f, total = M.start(), torch.zeros((len(doms), 2), dtype=F64, device=DEV)
    for _ in range(case["steps"]):
        f, B, rho, j = M.collide([f[q][src[q]] for q in range(9)], E)
        total += torch.stack([_body_sum(len(doms), dom, B * (j[0] - Fx)), _body_sum(len(doms), dom, B * j[1])], 1)
    return dict(drag=total / case["steps"])


def _exact_gradient(case, seed):
    """Reverse mode of the 64-bit steps: J = (1/T) sum over steps and cells of B j_x."""
    x, v, w, r = _disks(case, seed)
    size, n, N = (case["nx"], case["ny"]), len(r), case["steps"]
    body, cell, eps, arm = _disk_cells(x, r, size, (False, False))
    E = _solid_sums((size[1], size[0]), body, cell, eps, [0 * eps, 0 * eps])[0]
    M = _Model(size, case["tau"], 0.0, (0.0, 0.0), "inlet", "wall", case["u_in"])

    def step(f, E, u, tau):
        M.u_in = u
        g, B, rho, j = M.collide(M.pull(list(f)), E, None, tau)
        return torch.stack(g), (B * j[0]).sum() / N

    states, J = [torch.stack(M.start())], 0.0
    for _ in range(N):
        f, d = step(states[-1], E, case["u_in"], case["tau"])
        states.append(f)
        J = J + d
    lam, leaf = torch.zeros_like(states[0]), [E, torch.tensor(case["u_in"], dtype=F64, device=DEV), torch.tensor(case["tau"], dtype=F64, device=DEV)]
    acc = [torch.zeros_like(a) for a in leaf]
    for t in range(N - 1, -1, -1):
        args = [a.detach().requires_grad_() for a in (states[t], *leaf)]
        f, d = step(*args)
        g = torch.autograd.grad([f, d], args, [lam, torch.ones_like(d)])
        lam = g[0]
        if t == 0:   # f(0), pulled from the field the call starts from, is held fixed
            g = (g[0], g[1], 0.0, g[3])
        acc = [a + b for a, b in zip(acc, g[1:])]
    gE = acc[0].reshape(-1)[cell]
    x0, y0, rr = arm[0] - 0.5, arm[1] - 0.5, torch.as_tensor(r, dtype=F64, device=DEV)[body]

    def chord(a, lo):   # length of the disk's chord on the line at a within [lo, lo + 1]
        h = torch.sqrt((rr * rr - a * a).clamp(min=0))
        return (torch.minimum(lo + 1, h) - torch.maximum(lo, -h)).clamp(min=0) * (a.abs() < rr)
    gx = torch.stack([_body_sum(n, body, gE * (chord(x0, y0) - chord(x0 + 1, y0))),
                      _body_sum(n, body, gE * (chord(y0, x0) - chord(y0 + 1, x0)))], 1)
    return dict(J=J, duin=acc[1], dtau=acc[2], dx=gx)


def exact(case, seed):
    how = {"sweep": _exact_sweep, "gradient": _exact_gradient, "spheres": _exact_3d, "bed": _exact_3d}.get(case["kind"], _exact_2d)
    with torch.set_grad_enabled(case["kind"] == "gradient"):
        return how(case, seed)
