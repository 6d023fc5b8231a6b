"""What the library is measured on: runs as a user's program makes them.

A case is one call sequence of such a program on a lattice that it holds:
``steps`` time steps (``lb_step``) and the read-out that follows them, either
the fields (``lb_get_fields``) with the particle state or, in the runs that
follow the particles, the particle state alone (``lb_get_colloids``).  The
adjoint case is one evaluation of an objective and of its gradients.

Results are returned in the type that the lattice holds them in (the C ABI
widens all of them to FP64): FP64, FP32, or, for the fields of an FP16-storage
lattice and the velocities that its particles take from them, FP16; positions
and orientations of the particles of an FP16 lattice in FP32.

Inputs are seeded and synthetic: a noisy mixture with a large-scale velocity
field (the state of a run that is under way), and particles on a jittered
grid, moving with the fluid, some of them in contact.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2004_04080_gb300 import lbgb
from paper_2004_04080_gb300.adjoint import AdjointRunner, LBObjective
from paper_2004_04080_gb300.lbgb import LBLattice

BASE = dict(
    kind="mixture",    # "mixture" (two components), "single" (one component) or "adjoint"
    prec="fp32", nx=64, ny=64, nz=64,
    tau_a=1.0, tau_b=1.0,
    rho=1.0, noise=0.004,        # mean density of a component, relative standard deviation of its noise
    G=0.65, zeta=0.0,
    radius=0.0, particles=0, density=1.0,
    janus=False,       # Janus particles with lubrication and a pair list with a skin
    walls=False,       # walls normal to z moving at -+0.05 along x
    inlet=False,       # velocity inlet at the lower, pressure outlet at the upper z face, extrapolated
    steps=10,
    read="fields",     # "fields" (with the particle state) or "particles"
)


def _case(**kw):
    return dict(BASE, **kw)


def _filling(nx, ny, nz, radius, phi):
    return int(round(phi * nx * ny * nz / (4.0 / 3.0 * math.pi * radius ** 3)))


def listed():
    return [
        # the smallest call: a program that takes one step at a time and looks
        # at its particles after each (the 32^3 box of four particles)
        _case(name="small32_fp32_step", nx=32, ny=32, nz=32, rho=0.5, noise=0.006, radius=4.5, particles=4,
              steps=1, read="particles"),
        # the FP64 reference run of the same box, as the parity checks make it
        _case(name="small32_fp64", prec="fp64", nx=32, ny=32, nz=32, rho=0.5, noise=0.006, radius=4.5, particles=4,
              steps=20),
        # the bijel box in FP32: fields after a short run
        _case(name="bijel128_fp32", nx=128, ny=128, nz=128, radius=5.0, particles=801, steps=8),
        # the FP64 run that the reduced-precision forms are compared with
        _case(name="demix96_fp64", prec="fp64", nx=96, ny=96, nz=96, radius=5.0, particles=338, steps=10),
        # the confined bijel under shear at its full size, followed by its
        # (dense) particles
        _case(name="shear512_fp32", nx=512, ny=512, nz=256, rho=0.5, noise=0.006, radius=5.5, particles=14444,
              density=8.0, walls=True, steps=20, read="particles"),
        # the same run in FP16 storage on an eighth of the box
        _case(name="shear256_fp16", prec="fp16", nx=256, ny=256, nz=128, rho=0.5, noise=0.006, radius=5.5,
              particles=1806, density=8.0, walls=True, steps=12, read="particles"),
        # the colloid benchmark: Janus particles, lubrication, pair list with a skin
        _case(name="janus256_fp32", nx=256, ny=256, nz=256, zeta=0.1, radius=5.5, particles=2407, density=0.677,
              janus=True, steps=10, read="particles"),
        # the two-component benchmark without particles, one observation interval
        _case(name="case0_256_fp32", nx=256, ny=256, nz=256, steps=100),
        # the same mixture in FP16 storage, ragged sides, between moving walls
        _case(name="mixture_ragged_fp16", prec="fp16", nx=244, ny=150, nz=197, walls=True, steps=60),
        # the one-component benchmark, one observation interval
        _case(name="single256_fp32", kind="single", nx=256, ny=256, nz=256, noise=1e-4, steps=100),
        # unequal relaxation times: wetting particles in a channel with an
        # inlet and an outlet, ragged sides
        _case(name="channel_tau_fp32", nx=140, ny=92, nz=110, tau_a=0.8, tau_b=1.2, rho=0.5, noise=0.006, G=0.5,
              zeta=0.1, radius=4.5, particles=300, inlet=True, steps=8),
        # one gradient of drag and interface area: the adjoint box of eight
        # fixed particles with sqrt(N) checkpoints
        _case(name="adjoint64_fp32", kind="adjoint", nx=64, ny=64, nz=64, zeta=0.1, noise=0.03, radius=4.5,
              particles=8, steps=36, read="gradients"),
    ]


def draw(rng):
    def side(lo, hi, multiple=1):
        v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(lo, v // multiple * multiple)

    sort = rng.choice(["particles", "particles", "fields", "mixture", "mixture", "single", "tau", "adjoint"])
    if sort == "adjoint":
        n = [side(32, 72, 4), side(32, 72), side(32, 72)]
        return _case(kind="adjoint", nx=n[0], ny=n[1], nz=n[2], zeta=0.1, noise=0.03, radius=4.5,
                     particles=_filling(*n, 4.5, 0.011), steps=rng.randint(16, 36), read="gradients")
    prec = rng.choice(["fp32", "fp32", "fp16", "fp64"])
    if sort == "single":
        n = [side(24, 300, 4), side(24, 300), side(24, 300)]
        return _case(kind="single", prec=prec, nx=n[0], ny=n[1], nz=n[2], noise=1e-4, walls=rng.random() < 0.5,
                     tau_a=rng.choice([1.0, 1.0, 0.8]), steps=rng.randint(10, 40))
    if sort in ("mixture", "tau"):
        top = 240 if prec != "fp64" else 100
        n = [side(24, top, 4), side(24, top), side(24, top)]
        tau = (1.0, 1.0) if sort == "mixture" else rng.choice([(0.8, 1.2), (0.9, 0.9)])
        return _case(prec=prec, nx=n[0], ny=n[1], nz=n[2], walls=rng.random() < 0.5, tau_a=tau[0], tau_b=tau[1],
                     steps=rng.randint(10, 40))
    # particle runs: the fields after them only where few particles are followed
    if sort == "fields":
        prec = rng.choice(["fp32", "fp64"])
        n = [side(36, 110, 4), side(36, 110), side(36, 110)]
        return _case(prec=prec, nx=n[0], ny=n[1], nz=n[2], radius=rng.choice([4.5, 5.0]), zeta=rng.choice([0.0, 0.1]),
                     particles=max(1, _filling(*n, 5.0, rng.uniform(0.05, 0.2))), walls=rng.random() < 0.5,
                     tau_a=(t := rng.choice([1.0, 1.0, 0.9])), tau_b=t, steps=rng.randint(1, 8))
    prec = rng.choice(["fp32", "fp32", "fp16"])
    n = [side(48, 300, 4), side(48, 300), side(48, 300)]
    janus = rng.random() < 0.4
    return _case(prec=prec, nx=n[0], ny=n[1], nz=n[2], radius=5.5, particles=_filling(*n, 5.5, rng.uniform(0.05, 0.15)),
                 density=0.677 if janus else 8.0, rho=0.5, noise=0.006, walls=rng.random() < 0.5, janus=janus,
                 zeta=0.1 if janus else 0.0, steps=rng.randint(1, 8 if janus else 12), read="particles")


# ------------------------------------------------------------------ inputs
def _params(case):
    R = case["radius"]
    p = dict(tau=(case["tau_a"], case["tau_b"]), G=case["G"], rho0=(case["rho"], case["rho"]),
             zeta=(case["zeta"], -case["zeta"]))
    if case["kind"] == "single":
        p.update(tau=(case["tau_a"],) * 2, G=0.0, zeta=(0.0, 0.0))
    if case["kind"] == "adjoint":
        p.update(body_force=(2e-4, 0.0, 1e-4))
    if R:
        p.update(hertz_K=20.0, hertz_sigma=2 * R + 1.0, hertz_rcap=2 * R)
    if case["janus"]:
        p.update(zeta=(case["zeta"], case["zeta"]), janus=1, janus_theta0=108.0, janus_width=10.0, lub_on=1,
                 lub_scale=0.1, lub_hn=0.67, lub_hmin=0.5, rcut=2 * R + 1.0, delr=1.0)
    if case["walls"]:
        p.update(bc=(1, 1, 0), wall_u_lo=(-0.05, 0.0, 0.0), wall_u_hi=(0.05, 0.0, 0.0))
    if case["inlet"]:
        p.update(bc=(1, 1, 0), open=(2, 1), wall_u_lo=(0.0, 0.0, 0.02), open_rho=(case["rho"],) * 4, open_extrap=1)
    if R and not p.get("bc", (1, 1, 1))[2]:
        # (the interfaces of a demixing mixture push particles towards a wall)
        p.update(side_wall_k=1.0 if case["rho"] < 1.0 else 20.0, side_wall_d=R + 1.0)
    return p


def _generator(seed, what):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + what)


def _densities(case, seed):
    """rho^A, rho^B on the GPU, flat, FP64: m (1 + a eta) and m (1 - a eta)."""
    n = case["nx"] * case["ny"] * case["nz"]
    eta = torch.rand(n, generator=_generator(seed, 1), device="cuda", dtype=torch.float64) * 2 - 1
    eta *= case["noise"] * math.sqrt(3.0)
    a = case["rho"] * (1 + eta)
    b = torch.zeros_like(a) if case["kind"] == "single" else case["rho"] * (1 - eta)
    return a, b


def _velocity(case, x, y, z):
    """Large-scale velocity of the run at points (x, y, z): vortices across
    the box, on the shear profile of moving walls or the through-flow of an
    inlet."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    kx, ky = 2 * math.pi * x / nx, 2 * math.pi * y / ny
    bounded = case["walls"] or case["inlet"]
    sz = torch.sin(math.pi * (z + 0.5) / nz) if bounded else 0.6 + 0.4 * torch.cos(2 * math.pi * z / nz)
    ux = 0.03 * torch.sin(kx) * torch.cos(ky) * sz
    uy = -0.03 * torch.cos(kx) * torch.sin(ky) * sz
    uz = 0.01 * torch.sin(kx) * sz
    if case["walls"]:
        ux = ux + 0.1 * ((z + 0.5) / nz - 0.5)
    if case["inlet"]:
        uz = uz + 0.02
    return ux, uy, uz


def _velocity_field(case):
    g = [torch.arange(case[n], device="cuda", dtype=torch.float64) for n in ("nx", "ny", "nz")]
    z, y, x = torch.meshgrid(g[2], g[1], g[0], indexing="ij")
    return torch.stack([c.reshape(-1) for c in _velocity(case, x, y, z)])


def _particles(case, seed):
    """Particles on the points of a jittered grid: pos, vel, omega, quat (FP64, host)."""
    n, R = case["particles"], case["radius"]
    if not n:
        return None
    g = _generator(seed, 2)
    gap = R + 1.0 if case["walls"] or case["inlet"] else 0.0
    ext = [case["nx"], case["ny"], case["nz"] - 2 * gap]
    cells = [1, 1, 1]  # grid points per axis: the spacing grows until n points are left
    spacing = (float(np.prod(ext)) / n) ** (1 / 3)
    while int(np.prod(cells)) < n:
        cells = [max(1, int(e / spacing)) for e in ext]
        spacing *= 0.995
    step = [e / c for e, c in zip(ext, cells)]
    pick = torch.randperm(int(np.prod(cells)), generator=g, device="cuda")[:n]
    ix, iy, iz = pick % cells[0], pick // cells[0] % cells[1], pick // (cells[0] * cells[1])
    out = []
    for i, s, lo in ((ix, step[0], 0.0), (iy, step[1], 0.0), (iz, step[2], gap)):
        room = max(0.0, 0.5 * (s - 2 * R - 0.5))  # neighbours stay 2 R + 1/2 apart
        t = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
        out.append(lo + (i + 0.5) * s + t * room)
    pos = torch.stack(out, 1)
    if case["kind"] == "adjoint":
        return dict(pos=pos.cpu().numpy(), radius=np.full(n, R))
    vel = torch.stack(_velocity(case, *out), 1)
    omega = 0.01 * torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    quat = torch.randn((n, 4), generator=g, device="cuda", dtype=torch.float64)
    quat = quat / quat.norm(dim=1, keepdim=True)
    mass = case["density"] * 4.0 / 3.0 * math.pi * R ** 3
    return dict(pos=pos.cpu().numpy(), vel=vel.cpu().numpy(), omega=omega.cpu().numpy(), quat=quat.cpu().numpy(),
                radius=np.full(n, R), mass=np.full(n, mass))


def _theta(case):
    return [case["tau_a"], case["tau_b"], case["G"], case["zeta"], -case["zeta"]]


# --------------------------------------------------------------------- run
def prepare(case, seed):
    shape = (case["nx"], case["ny"], case["nz"])
    lat = LBLattice(shape, case["prec"], max_colloids=case["particles"],
                    components=1 if case["kind"] == "single" else 2)
    a, b = _densities(case, seed)
    parts = _particles(case, seed)
    state = dict(case=case, lat=lat)
    if case["kind"] == "adjoint":
        state.update(runner=AdjointRunner(lat, case["steps"]), particles=parts, params=_params(case),
                     theta=torch.tensor(_theta(case), dtype=torch.float32, requires_grad=True),
                     rho=[r.float().requires_grad_(True) for r in (a, b)])
        return state
    lat.set_params(**_params(case))
    single = case["kind"] == "single"
    lat.init_fields(a.cpu().numpy(), None if single else b.cpu().numpy(), _velocity_field(case).cpu().numpy())
    if parts is not None:
        lat.add_colloids(**parts)
    if case["read"] == "fields":  # the page-locked arrays that the program reads into, and where it keeps the values
        dtype = dict(fp64=torch.float64, fp32=torch.float32, fp16=torch.float16)[case["prec"]]
        state["host"] = [torch.empty((c, lat.N), dtype=torch.float64, pin_memory=True) for c in (1, 1, 3)]
        state["kept"] = {n: torch.zeros(h.shape, dtype=dtype) for n, h in zip(("rho_a", "rho_b", "u"), state["host"])}
        if single:
            del state["kept"]["rho_b"]
    return state


def _gradients(state):
    case, (ra, rb), theta = state["case"], state["rho"], state["theta"]
    p = {k: v for k, v in state["params"].items() if k not in ("tau", "G", "zeta")}
    value = LBObjective().apply(theta, ra, rb, state["runner"], p, state["particles"])
    grads = torch.autograd.grad(value[0] * 100.0 + value[1] / lat_sites(case), (theta, ra, rb))
    return dict(value=value.detach().float(), theta=grads[0], rho_a=grads[1], rho_b=grads[2])


def lat_sites(case):
    return case["nx"] * case["ny"] * case["nz"]


def run(state):
    case, lat = state["case"], state["lat"]
    if case["kind"] == "adjoint":
        return _gradients(state)
    lat.step(case["steps"])
    out = {}
    if case["read"] == "fields":
        host = dict(zip(("rho_a", "rho_b", "u"), state["host"]))
        lbgb.lb_get_fields(lat.h, *[h.numpy() for h in host.values()])
        out.update({n: t.copy_(host[n]) for n, t in state["kept"].items()})
    if case["particles"]:
        c = lat.get_colloids()
        place, rate = dict(fp64=(np.float64,) * 2, fp32=(np.float32,) * 2,
                           fp16=(np.float32, np.float16))[case["prec"]]
        out.update({k: c[k].astype(t) for k, t in (("pos", place), ("vel", rate), ("omega", rate), ("quat", place))})
    return out


def work(case):
    """Bytes and operations of one pass.  The populations come in and go out
    once.  In between, a step at tau = 1 needs the densities and the momentum
    of a site (f* is the equilibrium of these: Eq. 16 at omega = 1), a step
    at another tau its populations; reading the fields costs the FP64 values
    that go to the host."""
    n, s = lat_sites(case), case["steps"]
    store = dict(fp64=8, fp32=4, fp16=2)[case["prec"]]
    comp = 8 if case["prec"] == "fp64" else 4
    k = 1 if case["kind"] == "single" else 2
    unit = case["tau_a"] == 1.0 and (k == 1 or case["tau_b"] == 1.0)
    step_bytes = 2 * (k + 3) * comp if unit else 2 * 19 * k * store
    data = n * (2 * 19 * k * store + (s - 1) * step_bytes)
    flops = 200.0 * k * n * s
    if case["kind"] == "adjoint":  # forward, recomputation, and per step the state read and the adjoint field in and out
        data = n * (2 * s * step_bytes + s * 38 * (store + 2 * comp))
        flops *= 5
    elif case["read"] == "fields":
        data += 8 * n * (k + 3)
    return dict(bytes=float(data + 150 * 8 * case["particles"] * s), flops=flops)


# ------------------------------------------------------------------- exact
# The same run in FP64 with plain torch operations.
_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
      (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
      (0, -1, 1)]
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]


def _dot(c, v):
    """c . v for a link c and a list of three tensors (the zero terms left out)."""
    t = None
    for cd, vd in zip(c, v):
        if cd:
            x = vd if cd > 0 else -vd
            t = x if t is None else t + x
    return torch.zeros_like(v[0]) if t is None else t


def _equilibrium(i, rho, u, uu):
    cu = _dot(_C[i], u)
    return _W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)


def _shift(t, i):
    """t at x - c_i (periodic)."""
    c = _C[i]
    return torch.roll(t, (c[2], c[1], c[0]), (0, 1, 2)) if i else t


class _Exact:
    def __init__(self, case, theta=None):
        self.case, self.p = case, _params(case)
        if theta is not None:
            self.p.update(tau=(theta[0], theta[1]), G=theta[2], zeta=(theta[3], theta[4]))
        self.n = (case["nx"], case["ny"], case["nz"])
        self.nk = 1 if case["kind"] == "single" else 2
        self.wall = not self.p.get("bc", (1, 1, 1))[2]
        self.owner = None

    def init(self, rho, u):
        shape = self.n[::-1]
        rho = [r.reshape(shape) for r in rho[:self.nk]]
        u = [c.reshape(shape) for c in u]
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        return [[_equilibrium(i, r, u, uu) for i in range(19)] for r in rho]

    # ---- particles
    def add(self, parts):
        t = {k: torch.as_tensor(v, device="cuda", dtype=torch.float64) for k, v in parts.items()}
        self.np = len(t["pos"])
        self.pos, self.R = t["pos"], t["radius"]
        zero = torch.zeros_like(self.pos)
        self.mass = t.get("mass", torch.full_like(self.R, math.inf))
        self.vel, self.omg = t.get("vel", zero), t.get("omega", zero)
        self.quat = t.get("quat")
        self.prev = None
        self.owner = self.map()

    def map(self):
        own = torch.full(self.n[::-1], -1, device="cuda", dtype=torch.int64)
        m = int(math.ceil(float(self.R.max()))) + 1
        o = torch.arange(-m, m + 2, device="cuda")
        oz, oy, ox = (g.reshape(-1) for g in torch.meshgrid(o, o, o, indexing="ij"))
        off = torch.stack([ox, oy, oz], 1)
        for s in range(0, self.np, 2048):
            pos = self.pos[s:s + 2048]
            a = torch.floor(pos).long()[:, None, :] + off
            inside = ((a - pos[:, None, :]) ** 2).sum(2) < (self.R[s:s + 2048] ** 2)[:, None]
            if self.wall:
                inside &= (a[..., 2] >= 0) & (a[..., 2] < self.n[2])
            w, q = inside.nonzero(as_tuple=True)
            x, y, z = (a[w, q, d] % self.n[d] for d in range(3))
            own[z, y, x] = w + s
        return own

    def arm(self, idx, p):
        """x_s - r_p, minimum image, for nodes idx = (z, y, x) of particles p."""
        d = torch.stack([idx[2], idx[1], idx[0]], 1).double() - self.pos[p]
        for c in range(3):
            if c < 2 or not self.wall:
                d[:, c] -= self.n[c] * torch.round(d[:, c] / self.n[c])
        return d

    def add_terms(self, F, T, idx, p, f):
        F.index_add_(0, p, f)
        T.index_add_(0, p, torch.linalg.cross(self.arm(idx, p), f))

    def remap(self, f, F, T):
        new = self.map()
        old, self.owner = self.owner, new
        if torch.equal(old, new):
            return
        both = (old < 0) & (new < 0)
        idx = ((old < 0) & (new >= 0)).nonzero(as_tuple=True)
        rho, j = zip(*[self.moments([q[idx] for q in g]) for g in f])
        u, _ = self.mixture(rho, j)
        self.add_terms(F, T, idx, new[idx], (rho[0] + rho[1])[:, None] * torch.stack(u, 1))
        idx = ((old >= 0) & (new < 0)).nonzero(as_tuple=True)
        p = old[idx]
        num, den = [0.0, 0.0], 0.0
        for i in range(1, 19):
            c = _C[i]
            z = idx[0] + c[2]
            at = (z % self.n[2], (idx[1] + c[1]) % self.n[1], (idx[2] + c[0]) % self.n[0])
            ok = both[at] & ((z >= 0) & (z < self.n[2]) if self.wall else True)
            w = _W[i] * ok.double()
            for k in range(2):
                num[k] = num[k] + w * sum(q[at] for q in f[k])
            den = den + w
        d = self.arm(idx, p)
        uw = self.vel[p] + torch.linalg.cross(self.omg[p], d)
        ul = list(uw.unbind(1))
        uu = (uw ** 2).sum(1)
        total = 0.0
        for k in range(2):
            r = torch.where(den > 0, num[k] / den.clamp(min=1e-300), torch.full_like(den, self.p["rho0"][k]))
            for i in range(19):
                f[k][i][idx] = _equilibrium(i, r, ul, uu)
            total = total + r
        self.add_terms(F, T, idx, p, -total[:, None] * uw)

    def pair_forces(self):
        P, F = self.p, torch.zeros_like(self.pos)
        K, sg, cap = P["hertz_K"], P["hertz_sigma"], P["hertz_rcap"]
        nu = sum((t - 0.5) / 6.0 for t in P["tau"])
        for s in range(0, self.np, 1024):
            d = self.pos[None] - self.pos[s:s + 1024, None]
            for c in range(3):
                if c < 2 or not self.wall:
                    d[..., c] -= self.n[c] * torch.floor(d[..., c] / self.n[c] + 0.5)
            r = d.norm(dim=2)
            i, q = ((r < sg + 0.1) & (r > 0)).nonzero(as_tuple=True)
            d, r = d[i, q], r[i, q]
            h = d / r[:, None]
            mag = -2.5 * K * (sg - torch.clamp(r, min=cap)).clamp(min=0) ** 1.5 * (r < sg)
            if P.get("lub_on"):
                Ri, Rj = self.R[s + i], self.R[q]
                red = Ri * Rj / (Ri + Rj)
                gap = r - Ri - Rj
                vr = ((self.vel[s + i] - self.vel[q]) * h).sum(1)
                mag = mag - (6 * math.pi * nu * P["lub_scale"] * red ** 2 * vr * (gap < P["lub_hn"]) *
                             (1 / gap.clamp(min=P["lub_hmin"]) - 1 / P["lub_hn"]))
            F.index_add_(0, s + i, mag[:, None] * h)
        if P.get("side_wall_k"):
            lo, hi = self.pos[:, 2] + 0.5, self.n[2] - 0.5 - self.pos[:, 2]
            F[:, 2] += P["side_wall_k"] * ((P["side_wall_d"] - lo).clamp(min=0) - (P["side_wall_d"] - hi).clamp(min=0))
        return F

    def janus(self, p, d):
        q = self.quat[p]
        a, b, c, e = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        axis = torch.stack([a * a + b * b - c * c - e * e, 2 * (b * c + a * e), 2 * (b * e - a * c)], 1)
        ct = ((axis * d).sum(1) / d.norm(dim=1)).clamp(-1, 1)
        th, th0, w = torch.rad2deg(torch.arccos(ct)), self.p["janus_theta0"], self.p["janus_width"]
        t = ((th - th0 + 0.5 * w) / w).clamp(0, 1)
        return -1 + 2 * t * t * (3 - 2 * t)

    def integrate(self, Fl, Tl, F, T):
        Fp, Tp = self.prev if self.prev is not None else (Fl, Tl)
        self.prev = (Fl, Tl)
        F, T = F + 0.5 * (Fp + Fl), T + 0.5 * (Tp + Tl)
        self.vel = self.vel + F / self.mass[:, None]
        self.pos = self.pos + self.vel
        for c in range(3):
            if c < 2 or not self.wall:
                self.pos[:, c] %= self.n[c]
        w = self.omg + T / (0.4 * self.mass * self.R ** 2)[:, None]
        self.omg = w

        def rate(q):
            a, b, c, e = (q / q.norm(dim=1, keepdim=True)).unbind(1)
            rows = [[a * a + b * b - c * c - e * e, 2 * (b * c - a * e), 2 * (b * e + a * c)],
                    [2 * (b * c + a * e), a * a - b * b + c * c - e * e, 2 * (c * e - a * b)],
                    [2 * (b * e - a * c), 2 * (c * e + a * b), a * a - b * b - c * c + e * e]]
            x, y, z = (rows[0][d] * w[:, 0] + rows[1][d] * w[:, 1] + rows[2][d] * w[:, 2] for d in range(3))
            a, b, c, e = q.unbind(1)
            return 0.5 * torch.stack([-b * x - c * y - e * z, a * x - e * y + c * z, e * x + a * y - b * z,
                                      -c * x + b * y + a * z], 1)

        qd = rate(self.quat)
        for _ in range(20):
            qd = rate(self.quat + 0.5 * qd)
        q = self.quat + qd
        self.quat = q / q.norm(dim=1, keepdim=True)

    # ---- fluid
    def moments(self, f):
        rho = sum(f)
        j = []
        for d in range(3):
            t = 0.0
            for i in range(1, 19):
                if _C[i][d]:
                    t = t + f[i] if _C[i][d] > 0 else t - f[i]
            j.append(t)
        return rho, j

    def mixture(self, rho, j):
        om = [1 / t for t in self.p["tau"]]
        den = sum(o * r for o, r in zip(om, rho))
        u = [sum(o * q[d] for o, q in zip(om, j)) / den for d in range(3)]
        inv = sum(r * 3 / (t - 0.5) for r, t in zip(rho, self.p["tau"])) / sum(rho)
        return u, inv / (3 + 0.5 * inv)

    def wall_density(self, rho, solid):
        """The density beyond each wall: [side][k] planes."""
        out = []
        for side, z in ((0, 0), (1, self.n[2] - 1)):
            if self.p.get("open", (0, 0))[side] in (1, 3):
                out.append([torch.full_like(rho[0][0], self.p["open_rho"][2 * side + k]) for k in range(2)])
                continue
            fl = 1.0 - solid[z].double() if solid is not None else torch.ones_like(rho[0][0])
            num, den = [0.0, 0.0], 0.0
            for i in range(1, 19):
                if _C[i][2] != (1 if side == 0 else -1):
                    continue
                sh = ((-_C[i][1], -_C[i][0]), (0, 1))
                den = den + _W[i] * torch.roll(fl, *sh)
                for k in range(2):
                    num[k] = num[k] + _W[i] * torch.roll(fl * rho[k][z], *sh)
            out.append([torch.where(den > 0, num[k] / den.clamp(min=1e-300), 0 * den) for k in range(2)])
        return out

    def gradient(self, psi, beyond):
        """sum_i w_i psi(x + c_i) c_i of one component."""
        s = [0.0, 0.0, 0.0]
        for i in range(1, 19):
            t = _shift(psi, _OPP[i])
            if self.wall and _C[i][2]:
                side, z = (1, self.n[2] - 1) if _C[i][2] > 0 else (0, 0)
                edge = torch.roll(beyond[side], (-_C[i][1], -_C[i][0]), (0, 1))
                t = torch.cat([t[:z], edge[None]]) if z else torch.cat([edge[None], t[1:]])
            for d in range(3):
                if _C[i][d]:
                    s[d] = s[d] + (_W[i] * _C[i][d]) * t
        return s

    def forces(self, rho, F=None, T=None):
        """Shan-Chen and body forces of each component; the wetting force of
        the frontier nodes is added to F, T."""
        G = self.p["G"]
        g = self.p.get("body_force", (0.0, 0.0, 0.0))
        if self.nk == 1:
            return [[rho[0] * c for c in g]]
        solid = self.owner >= 0 if self.owner is not None else None
        beyond = self.wall_density(rho, solid) if self.wall else None
        psi = [torch.where(solid, 0.0, r) for r in rho] if solid is not None else rho
        if solid is not None:
            fl = (~solid).double()
            near = torch.zeros_like(solid)
            inb = torch.arange(self.n[2], device="cuda")[:, None, None]
            for i in range(1, 19):
                t = _shift(~solid, i)
                if self.wall and _C[i][2]:
                    t = t & (inb != (0 if _C[i][2] > 0 else self.n[2] - 1))
                near |= t
            idx = (solid & near).nonzero(as_tuple=True)
            p = self.owner[idx]
            num, den, S = [0.0, 0.0], 0.0, [[0.0] * 3, [0.0] * 3]
            for i in range(1, 19):
                c = _C[i]
                z = idx[0] + c[2]
                at = (z % self.n[2], (idx[1] + c[1]) % self.n[1], (idx[2] + c[0]) % self.n[0])
                w = _W[i] * fl[at]
                if self.wall:
                    w = w * ((z >= 0) & (z < self.n[2]))
                den = den + w
                for k in range(2):
                    t = w * psi[k][at]
                    num[k] = num[k] + t
                    S[k] = [s + c[d] * t for d, s in enumerate(S[k])]
            zeta = self.p["zeta"]
            fac = [1 + zeta[0], 1 + zeta[1]]
            if self.p.get("janus"):
                sw = self.janus(p, self.arm(idx, p))
                fac = [1 + sw * zeta[0], 1 - sw * zeta[1]]
            v = [fac[k] * num[k] / den for k in range(2)]
            psi = [q.index_put(idx, t) for q, t in zip(psi, v)]
            if F is not None:
                self.add_terms(F, T, idx, p, torch.stack([-G * (v[0] * S[1][d] + v[1] * S[0][d]) for d in range(3)], 1))
        S = [self.gradient(psi[k], [b[k] for b in beyond] if beyond else None) for k in range(2)]
        return [[rho[k] * (g[d] - G * S[1 - k][d]) for d in range(3)] for k in range(2)]

    def face(self, f, rho, u, k, i, z, fs):
        """The population that comes back from the z face beyond link i, on
        the plane z: walls and velocity faces (Eq. 9), pressure faces (Eq. 10)."""
        side = 0 if z == 0 else 1
        kind = self.p.get("open", (0, 0))[side]
        zi = 1 if side == 0 else self.n[2] - 2
        ok = None if self.owner is None else self.owner[zi] < 0

        def out(q):
            e = 0.5 * (q[z] - q[zi])
            return q[z] + (e if ok is None else torch.where(ok, e, 0 * e))

        ext = self.p.get("open_extrap")
        if kind == 1:
            uw = [out(c) for c in u] if ext else [c[z] for c in u]
            cu = _dot(_C[i], uw)
            uu = uw[0] ** 2 + uw[1] ** 2 + uw[2] ** 2
            return -fs[z] + 2 * _W[i] * self.p["open_rho"][2 * side + k] * (1 + 4.5 * cu * cu - 1.5 * uu)
        uw = self.p.get("wall_u_lo" if side == 0 else "wall_u_hi", (0.0, 0.0, 0.0))
        rw = out(rho[k]) if kind == 2 and ext else rho[k][z]
        return fs[z] - 6 * _W[i] * rw * sum(c * v for c, v in zip(_C[i], uw))

    def step(self, f):
        """f(t) -> f(t + 1) (lists [k][i]); moves the particles; returns also F_liq."""
        moving = self.owner is not None and bool(torch.isfinite(self.mass).any())
        F = T = None
        if self.owner is not None:
            F, T = torch.zeros_like(self.pos), torch.zeros_like(self.pos)
        if moving:
            self.remap(f, F, T)
            F = F + self.pair_forces()
        rho, j = zip(*[self.moments(g) for g in f])
        solid = None
        if self.owner is not None:
            solid = self.owner >= 0
            rho = [torch.where(solid, r0, r) for r, r0 in zip(rho, self.p["rho0"])]
            j = [[torch.where(solid, 0.0, q) for q in g] for g in j]
        force = self.forces(rho, F if moving else None, T)
        if self.nk == 1:
            u, om = [q / rho[0] for q in j[0]], 1 / self.p["tau"][0]
        else:
            u, om = self.mixture(rho, j)
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        new = [[None] * 19 for _ in f]
        Fl = torch.zeros_like(self.pos) if self.owner is not None else None
        Tl = torch.zeros_like(self.pos) if self.owner is not None else None
        plain = not torch.is_tensor(self.p["tau"][0]) and all(t == 1.0 for t in self.p["tau"])
        for k, g in enumerate(f):
            us = [u[d] + force[k][d] / rho[k] for d in range(3)]
            uus = us[0] ** 2 + us[1] ** 2 + us[2] ** 2

            def star(i):
                e = _equilibrium(i, rho[k], us, uus)
                return e if plain else (1 - om) * (g[i] - _equilibrium(i, rho[k], u, uu)) + e

            new[k][0] = star(0)
            for i in range(1, 19, 2):
                pair = [star(i), star(i + 1)]
                for a, (l, o) in enumerate(((i, i + 1), (i + 1, i))):
                    # plane l of the new state: pushed along c_l, or bounced
                    # off a particle or a face reached along c_o
                    t = _shift(pair[a], l)
                    if solid is not None:
                        hit = _shift(solid, l) & ~solid
                        if self.wall and _C[l][2]:
                            hit[0 if _C[l][2] > 0 else -1] = False
                        idx = hit.nonzero(as_tuple=True)
                        c = _C[o]
                        p = self.owner[(idx[0] + c[2]) % self.n[2], (idx[1] + c[1]) % self.n[1],
                                       (idx[2] + c[0]) % self.n[0]]
                        uw = self.vel[p] + torch.linalg.cross(self.omg[p], self.arm(idx, p))
                        cw = uw @ torch.tensor(c, device="cuda", dtype=torch.float64)
                        out = pair[1 - a][idx]
                        back = out - 6 * _W[l] * rho[k][idx] * cw
                        t = t.index_put(idx, back)
                        fl = (out + back)[:, None] * torch.tensor(c, device="cuda", dtype=torch.float64)
                        Fl = Fl.index_add(0, p, fl)
                        Tl = Tl.index_add(0, p, torch.linalg.cross(self.arm(idx, p), fl))
                    if self.wall and _C[l][2]:
                        z = 0 if _C[l][2] > 0 else self.n[2] - 1
                        edge = self.face(f, rho, u, k, o, z, pair[1 - a])[None]
                        if solid is not None:
                            edge = torch.where(solid[z], 0.0, edge)
                        t = torch.cat([edge, t[1:]]) if z == 0 else torch.cat([t[:-1], edge])
                    new[k][l] = t
        if moving:
            self.integrate(Fl, Tl, F, T)
        return new, Fl

    def fields(self, f):
        rho, j = zip(*[self.moments(g) for g in f])
        force = self.forces(list(rho))
        u = [sum(q[d] + 0.5 * c[d] for q, c in zip(j, force)) / sum(rho) for d in range(3)]
        out = list(rho) + u
        if self.owner is not None:
            out = [torch.where(self.owner >= 0, 0.0, q) for q in out]
        out = [q.reshape(1, -1) for q in out]
        return out[:self.nk] + [torch.cat(out[self.nk:])]


def exact(case, seed):
    if lat_sites(case) * case["steps"] > 2.5e9:
        return None  # over a fraction of a minute
    a, b = _densities(case, seed)
    parts = _particles(case, seed)
    if case["kind"] == "adjoint":
        return _exact_gradients(case, a.float().double(), b.float().double(), parts)
    with torch.no_grad():
        e = _Exact(case)
        f = e.init([a, b], _velocity_field(case))
        del a, b
        if parts is not None:
            e.add(parts)
        for _ in range(case["steps"]):
            f, _ = e.step(f)
        out = {}
        if case["read"] == "fields":
            # (particles after the last step have moved: the fields are read on the last node map)
            names = ("rho_a", "rho_b", "u") if e.nk == 2 else ("rho_a", "u")
            out.update(zip(names, e.fields(f)))
        if parts is not None:
            out.update({k: v.cpu().numpy() for k, v in
                        dict(pos=e.pos, vel=e.vel, omega=e.omg, quat=e.quat).items()})
        return out


def _exact_gradients(case, a, b, parts):
    from torch.utils.checkpoint import checkpoint

    theta = torch.tensor(_theta(case), dtype=torch.float32, device="cuda").double().requires_grad_(True)
    a.requires_grad_(True)
    b.requires_grad_(True)
    e = _Exact(case, theta.unbind())
    e.add(parts)
    f = e.init([a, b], torch.zeros((3, lat_sites(case)), device="cuda", dtype=torch.float64))
    drag = 0.0

    def one(*flat):
        new, Fl = e.step([list(flat[:19]), list(flat[19:])])
        return (*new[0], *new[1], torch.sqrt((Fl ** 2).sum(1) + 1e-24).mean())

    for _ in range(case["steps"]):
        *flat, d = checkpoint(one, *f[0], *f[1], use_reentrant=False)
        f = [flat[:19], flat[19:]]
        drag = drag + d / case["steps"]
    fluid = e.owner < 0
    rho = [sum(g)[fluid] for g in f]
    phi = (rho[0] - rho[1]) / (rho[0] + rho[1])
    area = (1 - phi ** 2).sum()
    grads = torch.autograd.grad(drag * 100.0 + area / lat_sites(case), (theta, a, b))
    return dict(value=torch.stack([drag, area]).detach(), theta=grads[0], rho_a=grads[1], rho_b=grads[2])
