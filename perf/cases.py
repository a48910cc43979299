"""Performance cases of the lbsc framework: what its users have it do, through its public entry points.

A case is a dict of plain values; ``prepare`` makes what a user's program has in hand before the call, ``run``
is one pass through the public API, ``work`` the bytes and operations the pass cannot do without, ``exact`` the
same outputs in 64 bits by plain torch. Sizes are those of the repository's benchmark workloads and tests
(32^3 ... 256x256x128), or generic odd ones.

Kinds of case:
  step     a droplet (on a wall, free in a periodic box, or on a wall with posts) advanced by a number of steps,
           then its densities read back: the simulation itself, in every storage precision
  sweep    droplets of several box sizes and parameters advanced together as one Batch, then measured
  adjoint  the gradient of the droplet's height with respect to the wall parameters, with the final densities
  observe  the measurements between two runs: conservation sums and the contact angle at three levels
  tension  planar and radial surface tension of a state
  search   one iteration of a parameter search: new wall parameter, new initial state, a short run, the angle
           and every macroscopic field
  sums     FP64 conservation sums of a device population array (the allocation-free entry point)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0910_3915_gb300 import lbsc

CONTACT = dict(g_br=0.08, force_weights=1, force_scale=1.25)  # the droplet-forming parameter set of the benchmark
BYTES = {"f32": 304, "f16": 152, "bf16": 152}  # a node update: 38 populations read once and written once
FLOPS_PER_UPDATE = 800


def listed():
    return [
        # the smallest lattice of the repository's workloads, a run between two readbacks: launches and latency count
        dict(name="droplet-32", kind="step", nx=32, ny=32, nz=32, precision="f32", geometry="walls", tau_r=1.0, tau_b=1.0,
             steps=400),
        # the repository's main workload
        dict(name="droplet-128", kind="step", nx=128, ny=128, nz=128, precision="f32", geometry="walls", tau_r=1.0,
             tau_b=1.0, steps=500),
        # the 16-bit storage workload, the largest lattice of the default benchmark line
        dict(name="droplet-256-bf16", kind="step", nx=256, ny=256, nz=128, precision="bf16", geometry="walls", tau_r=1.0,
             tau_b=1.0, steps=300),
        # the other 16-bit format, with odd edges that no tile divides
        dict(name="droplet-odd-f16", kind="step", nx=201, ny=147, nz=75, precision="f16", geometry="walls", tau_r=1.0,
             tau_b=1.0, steps=300),
        # components of unequal viscosity, odd edges: every population enters the collision
        dict(name="viscosities-odd", kind="step", nx=90, ny=70, nz=53, precision="f32", geometry="walls", tau_r=0.9,
             tau_b=1.2, steps=300),
        # the free droplet of the surface-tension workload: a mask geometry, periodic along z too
        dict(name="free-drop-64", kind="step", nx=64, ny=64, nz=64, precision="f32", geometry="periodic", tau_r=1.0,
             tau_b=1.0, steps=400),
        # a parameter sweep in boxes of the sweep workload's edges
        dict(name="sweep-12", kind="sweep", boxes=12, draw=3, precision="f32", steps=150),
        # the calibration workload's lattice and checkpoint distance
        dict(name="adjoint-64", kind="adjoint", nx=64, ny=64, nz=64, tau_r=1.0, tau_b=1.0, steps=300, ckpt=100),
        # what is measured between two runs at the main workload's size
        dict(name="observe-128", kind="observe", nx=128, ny=128, nz=128, precision="f32"),
        # surface tensions of the sessile droplet of the surface-tension workload
        dict(name="tension-96", kind="tension", nx=96, ny=96, nz=96, precision="f32"),
        # one iteration of the search for a wall parameter
        dict(name="search-64", kind="search", nx=64, ny=64, nz=64, precision="f32", steps=100),
        # conservation sums for a caller that may not allocate
        dict(name="sums-64", kind="sums", nx=64, ny=64, nz=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "sweep", "adjoint", "observe", "tension", "search", "sums"])
    if kind == "step":
        precision = rng.choice(["f32", "f32", "f16", "bf16"])
        geometry = rng.choice(["walls", "walls", "walls", "periodic", "posts"])
        nx, ny, nz = _log(rng, 20, 256), _log(rng, 20, 256), _log(rng, 16, 128)
        tau_r, tau_b = rng.choice([(1.0, 1.0), (1.0, 1.0), (round(rng.uniform(0.85, 1.0), 3), round(rng.uniform(1.0, 1.2), 3))])
        steps = max(40, min(400, int(3e8 / (nx * ny * nz)))) + rng.randrange(32)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, geometry=geometry, tau_r=tau_r, tau_b=tau_b,
                    steps=steps)
    if kind == "sweep":
        return dict(kind=kind, boxes=rng.randrange(3, 15), draw=rng.randrange(1000), precision=rng.choice(["f32", "f32", "bf16"]),
                    steps=rng.randrange(60, 150))
    nx, ny, nz = _log(rng, 24, 128), _log(rng, 24, 128), _log(rng, 24, 128)
    if kind == "adjoint":
        nx, ny, nz = min(nx, 72), min(ny, 72), min(nz, 64)
        tau_r, tau_b = rng.choice([(1.0, 1.0), (1.0, 1.0), (0.9, 1.1)])
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, tau_r=tau_r, tau_b=tau_b, steps=rng.randrange(40, 200), ckpt=rng.choice([20, 50, 100]))
    if kind == "sums":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz)
    precision = rng.choice(["f32", "f32", "f16", "bf16"])
    if kind == "search":
        nx, ny, nz = min(nx, 96), min(ny, 96), min(nz, 96)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, steps=rng.randrange(40, 200))
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision)


# ---------------------------------------------------------------- inputs

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _fields(nx, ny, nz, seed, centre, radius, smooth=0.0):
    """Densities of a droplet 0.7 / 0.04 with +-1e-3 noise, as workloads.droplet_fields makes them; smooth > 0 gives the
    tanh profile of a relaxed interface instead of the initial step."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(1000003 * (seed % 100000) + nx + 7 * ny + 49 * nz)
    radius = radius * (1.0 + 0.04 * float(torch.rand(1, generator=g, device=dev, dtype=torch.float64) - 0.5))
    z, y, x = torch.meshgrid(*(torch.arange(n, device=dev, dtype=torch.float64) for n in (nz, ny, nx)), indexing="ij")
    d = torch.sqrt((x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2)
    s = torch.tanh((radius - d) / smooth) if smooth else torch.where(d <= radius, 1.0, -1.0).to(torch.float64)
    noise = (torch.rand((2, nz, ny, nx), generator=g, device=dev, dtype=torch.float64) - 0.5) * 2e-3
    return 0.37 + 0.33 * s + noise[0], 0.37 - 0.33 * s + noise[1]


def _sessile(case, seed, smooth=0.0):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    return _fields(nx, ny, nz, seed, (nx / 2, ny / 2, 0.5), 0.26 * min(nx, ny, 1.4 * nz), smooth)


def _step_fields(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["geometry"] == "periodic":
        return _fields(nx, ny, nz, seed, (nx / 2, ny / 2, nz / 2), 0.25 * min(nx, ny, nz))
    return _sessile(case, seed)


def _solid(case):
    """uint8 mask (nz, ny, nx): planar walls, none, or planar walls with square posts on the bottom one."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    s = np.zeros((nz, ny, nx), np.uint8)
    if case.get("geometry", "walls") != "periodic":
        s[0] = s[-1] = 1
    if case.get("geometry") == "posts":
        px, py = (np.arange(nx) % 10) < 4, (np.arange(ny) % 10) < 4
        s[1:4] |= (py[:, None] & px[None, :]).astype(np.uint8)
    return s


def _params(case, w=0.05):
    return dict(CONTACT, tau_r=case.get("tau_r", 1.0), tau_b=case.get("tau_b", 1.0), eta_wall_r=-w, eta_wall_b=w)


def _boxes(case):
    r = np.random.Generator(np.random.PCG64(case["draw"]))
    edges = r.choice(np.array([48, 64, 80, 96]), size=case["boxes"])
    g, w = r.uniform(0.07, 0.09, size=case["boxes"]), r.uniform(-0.1, 0.1, size=case["boxes"])
    return [(int(e), dict(CONTACT, g_br=float(a), tau_r=1.0, tau_b=1.0, eta_wall_r=-float(b), eta_wall_b=float(b)))
            for e, a, b in zip(edges, g, w)]


def _host(t):
    return t.cpu().numpy()


# ---------------------------------------------------------------- the passes

def prepare(case, seed):
    kind = case["kind"]
    if kind == "sums":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        n = 0.01 + 0.05 * torch.rand((2, 19, nz, ny, nx), generator=g, device="cuda", dtype=torch.float64)
        return dict(case=case, n=n, solid=torch.from_numpy(_solid(case)).cuda(), cons=torch.zeros(8, device="cuda", dtype=torch.float64))
    if kind == "sweep":
        boxes = _boxes(case)
        fields = [tuple(map(_host, _sessile(dict(nx=e, ny=e, nz=e), seed + 31 * i))) for i, (e, _) in enumerate(boxes)]
        return dict(case=case, batch=lbsc.Batch(fields, [lbsc.Params(**p) for _, p in boxes], case["precision"]))
    if kind == "step":
        rr, rb = map(_host, _step_fields(case, seed))
    else:
        rr, rb = map(_host, _sessile(case, seed, smooth=2.5 if kind in ("observe", "tension") else 0.0))
    lat = lbsc.Lattice(rr, rb, case.get("precision", "f32"))
    if case.get("geometry", "walls") != "walls":
        lat.set_geometry(_solid(case))
    lat.set_params(**_params(case))
    if kind == "tension":
        lat.step(20)
    state = dict(case=case, lat=lat)
    if kind == "search":
        state.update(rr=rr, rb=rb, tries=0)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sums":
        lbsc.conservation_static(state["n"].data_ptr(), state["solid"].data_ptr(), case["nx"], case["ny"], case["nz"],
                                 state["cons"].data_ptr())
        return state["cons"]
    if kind == "sweep":
        b = state["batch"]
        b.step(case["steps"])
        angles, cons = b.contact_angles(5.0), b.conservation()
        return dict(cons=cons, rho=[b.box(i).moments()[:2] for i in range(b.n)], theta=[a["theta_deg"] for a in angles],
                    theta_fit=[a["theta_fit_deg"] for a in angles])
    lat = state["lat"]
    if kind == "step":
        lat.step(case["steps"])
        rr, rb, _, cons = lat.moments()
        return dict(rho_r=rr, rho_b=rb, cons=cons)
    if kind == "adjoint":
        J, g = lat.step_backward(case["steps"], case["ckpt"], "com_soft")
        rr, rb, _, cons = lat.moments()
        return dict(J=J, g=g, rho_r=rr, rho_b=rb, cons=cons)
    if kind == "observe":
        cons, zero = lat.measure(5.0)
        high = lat.contact_angle(5.0, level=0.5 * zero["phi_max"])
        low = lat.contact_angle(5.0, level=0.5 * zero["phi_min"])
        return dict(cons=cons, zero=zero, high=high, low=low)
    if kind == "tension":
        prof, gsum = lat.pressure_profile()
        bins, gamma, rs = lat.pressure_radial(_centre(case), 1.0, 2 * case["nz"], 5.5, case["nz"] / 2 - 5)
        return dict(prof=prof, gsum=gsum, bins=bins, gamma=gamma, R_s=rs)
    # search: another wall parameter in every iteration
    lat.set_params(**_params(case, 0.05 - 0.02 * (state["tries"] % 4)))
    state["tries"] += 1
    lat.reset(state["rr"], state["rb"])
    lat.step(case["steps"])
    drop = lat.contact_angle(5.0)
    rr, rb, u, cons = lat.moments(velocity=True)
    return dict(drop=drop, rho_r=rr, rho_b=rb, u=u, cons=cons)


def _centre(case):
    return case["nx"] / 2, case["ny"] / 2, 0.5


def _fluid(case):
    return int((_solid(case) == 0).sum())


def work(case):
    kind = case["kind"]
    if kind == "sums":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 305 * n + 64, "flops": 38 * 4 * n}
    if kind == "sweep":
        n = sum(e * e * (e - 2) for e, _ in _boxes(case))
        updates = n * case["steps"]
        return {"bytes": updates * BYTES[case["precision"]] + n * (BYTES[case["precision"]] // 2 + 16), "flops": updates * FLOPS_PER_UPDATE}
    n = _fluid(case)
    state = BYTES[case.get("precision", "f32")] // 2
    if kind == "step":
        return {"bytes": n * (case["steps"] * 2 * state + state + 16), "flops": n * case["steps"] * FLOPS_PER_UPDATE}
    if kind == "adjoint":
        # the forward run, the recompute, and per reverse step one read of the state and one of the adjoint's 8 fields
        # each way (at tau = 1; the 38 populations otherwise)
        adj = 64 if case["tau_r"] == case["tau_b"] == 1.0 else 304
        return {"bytes": n * (case["steps"] * (4 * state + state + adj) + state + 16), "flops": n * case["steps"] * 4 * FLOPS_PER_UPDATE}
    if kind == "observe":
        return {"bytes": n * state, "flops": n * 150}
    if kind == "tension":
        return {"bytes": 2 * n * state, "flops": n * 1200}
    return {"bytes": n * (16 + case["steps"] * 2 * state + state + 40), "flops": n * case["steps"] * FLOPS_PER_UPDATE}


# ---------------------------------------------------------------- the same in 64 bits, by plain torch

C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
     (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
Z = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
OPP = [0] + [k + 1 if k % 2 else k - 1 for k in range(1, 19)]


def _roll(a, c):
    """a at x - c: the value moved along +c (the last three axes are z, y, x)."""
    return torch.roll(a, (c[2], c[1], c[0]), (-3, -2, -1)) if any(c) else a


def _dot(c, v):
    """c . v for a velocity of entries -1, 0, 1 (v: three arrays)."""
    out = None
    for s, a in zip(c, v):
        if s:
            out = (a if s > 0 else -a) if out is None else (out + a if s > 0 else out - a)
    return out


class _Exact:
    """The method in 64 bits: populations n (2, 19, nz, ny, nx)."""

    def __init__(self, solid, p):
        self.solid = torch.from_numpy(solid).to(_device()).bool()
        self.from_wall = [_roll(self.solid, c) for c in C]  # x - c is solid
        self.p = p
        self.G = [0.0] + [(2.0 if k <= 6 else 1.0) if p["force_weights"] else 1.0 for k in range(1, 19)]
        self.gk = p["g_br"] * p["force_scale"]
        self.eta = torch.tensor([p["eta_wall_r"], p["eta_wall_b"]], dtype=torch.float64, device=_device())

    def rest(self, rr, rb):
        r = torch.stack([rr, rb]) * ~self.solid
        return torch.stack([z * r for z in Z], 1)

    def moments(self, n):
        rho = n.sum(1)
        j = [sum(C[k][d] * n[:, k] for k in range(19) if C[k][d]) for d in range(3)]
        return rho, j

    def psi(self, rho, eta):
        return torch.where(self.solid, eta[:, None, None, None], -torch.expm1(-rho))

    def force(self, psi):
        """(2, ...) arrays along x, y, z."""
        S = [0.0, 0.0, 0.0]
        other = psi.flip(0)
        for k in range(1, 19):
            v = self.G[k] * _roll(other, tuple(-c for c in C[k]))
            for d in range(3):
                if C[k][d]:
                    S[d] = S[d] + C[k][d] * v
        return [-self.gk * psi * s for s in S]

    def step(self, n, eta=None):
        eta = self.eta if eta is None else eta
        t = torch.tensor([self.p["tau_r"], self.p["tau_b"]], dtype=n.dtype, device=n.device)[:, None, None, None]
        rho, j = self.moments(n)
        F = self.force(self.psi(rho, eta))
        safe = torch.where(self.solid, 1.0, rho)
        den = (safe / t).sum(0)
        u = [(j[d] / t).sum(0) / den + t * F[d] / safe for d in range(3)]
        usq = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        post = []
        for k in range(19):
            cu = _dot(C[k], u)
            q = Z[k] * rho * (1 - 1.5 * usq if cu is None else 1 + cu * (3 - 4.5 * usq + 4.5 * cu * (1 + cu)) - 1.5 * usq)
            post.append(q if self.p["tau_r"] == self.p["tau_b"] == 1.0 else n[:, k] + (q - n[:, k]) / t)
        out = [torch.where(self.from_wall[k], post[OPP[k]], _roll(post[k], C[k])) for k in range(19)]
        return torch.stack(out, 1) * ~self.solid

    def velocity(self, n):
        rho, j = self.moments(n)
        F = self.force(self.psi(rho, self.eta))
        tot = torch.where(self.solid, 1.0, rho.sum(0))
        return torch.stack([torch.where(self.solid, 0.0, (j[d].sum(0) + 0.5 * F[d].sum(0)) / tot) for d in range(3)])

    def cons(self, n, steps):
        rho, j = self.moments(n)
        return torch.stack([rho[0].sum(), rho[1].sum(), *(a.sum() for a in j), torch.zeros((), device=n.device),
                            (~self.solid).sum().double(), torch.full((), float(steps), device=n.device)])


def _droplet(phi, solid, offset, level):
    """The droplet record of phi = rho_r - rho_b (whole-number entries None), planar walls."""
    f = phi - level
    nz = phi.shape[0]
    zw, zref = 0.5, 0.5 + offset
    pts, top = [], -math.inf
    for d, ax in ((0, 2), (1, 1), (2, 0)):
        lo = [slice(None)] * 3
        hi = [slice(None)] * 3
        lo[ax], hi[ax] = slice(0, -1), slice(1, None)
        q0, q1 = f[tuple(lo)], f[tuple(hi)]
        cross = ((q0 > 0) != (q1 > 0)) & ~solid[tuple(lo)] & ~solid[tuple(hi)]
        at = torch.nonzero(cross)
        a, b = q0[cross], q1[cross]
        t = a / (a - b)
        p = at.flip(1).double()  # x, y, z
        p[:, d] += t
        if d == 2 and len(a):
            up = p[a > 0, 2]
            top = float(up.max()) if len(up) else top
        pts.append(p[p[:, 2] >= zref])
    pts = torch.cat(pts)
    fl = phi[~solid]
    out = dict(phi_max=float(fl.max()), phi_min=float(fl.min()), h=top - zw, ok=None, status=None, n_points=None)
    z0 = int(math.floor(zref))
    bref = 0.0
    if z0 + 1 < nz:
        fz = zref - z0
        a0 = (1 - fz) * f[z0] + fz * f[z0 + 1]
        a1 = torch.roll(a0, -1, 1)
        part = torch.where(a0 > 0, a0 / (a0 - a1), a1 / (a1 - a0))
        length = torch.where((a0 > 0) & (a1 > 0), 1.0, torch.where((a0 <= 0) & (a1 <= 0), 0.0, part))
        bref = 2 * math.sqrt(float(length.sum()) / math.pi)
    out["base_ref"] = bref
    h, hp = out["h"], out["h"] - offset
    out.update(theta_deg=0.0, theta_fit_deg=0.0, b=0.0, r=0.0, xc=0.0, yc=0.0, zc=0.0, r_fit=0.0)
    if z0 + 1 < nz and math.isfinite(top) and hp > 0 and bref > 0:
        r = (0.25 * bref * bref + hp * hp) / (2 * hp)
        b = 2 * math.sqrt(max(r * r - (r - h) ** 2, 0.0))
        out.update(r=r, b=b, theta_deg=math.degrees(math.atan2(0.5 * b, r - h)))
    if len(pts) >= 4:
        A = torch.cat([2 * pts, torch.ones_like(pts[:, :1])], 1)
        s = torch.linalg.solve(A.T @ A, A.T @ (pts ** 2).sum(1)).tolist()
        R = math.sqrt(s[3] + s[0] ** 2 + s[1] ** 2 + s[2] ** 2)
        out.update(xc=s[0], yc=s[1], zc=s[2], r_fit=R, theta_fit_deg=math.degrees(math.acos(max(-1.0, min(1.0, -(s[2] - zw) / R)))))
    if not math.isfinite(out["h"]):
        out["h"] = None
    return out


def _tension(ex, n, case):
    """Plane means and radial bins of the pressure tensor."""
    rho, _ = ex.moments(n)
    u = ex.velocity(n)
    psi = ex.psi(rho, ex.eta)
    pairs = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]
    P = [torch.zeros_like(rho[0]) for _ in pairs]
    for k in range(19):
        m = n[:, k].sum(0)
        v = [C[k][d] - u[d] for d in range(3)]
        w = 0.0
        if k:
            o = [_roll(psi[a], tuple(-c for c in C[k])) for a in (0, 1)]
            w = 0.5 * ex.gk * ex.G[k] * (psi[0] * o[1] + psi[1] * o[0])
        for i, (a, b) in enumerate(pairs):
            P[i] += v[a] * v[b] * m + (w * C[k][a] * C[k][b] if k else 0.0)
    fluid = (~ex.solid).double()
    phi = rho[0] - rho[1]
    cnt = fluid.sum((1, 2))
    prof = torch.stack([(v * fluid).sum((1, 2)) / cnt.clamp(min=1) for v in (*P, phi)] + [cnt], 1)
    gsum = float(torch.where(cnt > 0, prof[:, 2] - 0.5 * (prof[:, 0] + prof[:, 1]), 0.0).sum())
    nz, ny, nx = phi.shape
    c = _centre(case)
    z, y, x = torch.meshgrid(*(torch.arange(m, device=phi.device, dtype=torch.float64) for m in (nz, ny, nx)), indexing="ij")
    d = [x - c[0], y - c[1], z - c[2]]
    d[0] = d[0] - nx * torch.round(d[0] / nx)
    d[1] = d[1] - ny * torch.round(d[1] / ny)
    r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    nb, zmin, rmax = 2 * nz, 5.5, nz / 2 - 5
    take = (~ex.solid) & (z >= zmin) & (r > 0) & (torch.floor(r) < nb)
    e = [a / torch.where(r > 0, r, 1.0) for a in d]
    pn = sum((1.0 if a == b else 2.0) * e[a] * e[b] * P[i] for i, (a, b) in enumerate(pairs))
    pt = 0.5 * (P[0] + P[1] + P[2] - pn)
    idx = torch.floor(r[take]).long()
    bins = torch.zeros((nb, 4), dtype=torch.float64, device=phi.device)
    for v, a in enumerate((pn, pt, phi, torch.ones_like(phi))):
        bins[:, v].index_add_(0, idx, a[take])
    bins[:, :3] /= bins[:, 3:].clamp(min=1)
    B = bins.tolist()
    rs, prev = math.nan, None
    for b in range(nb):
        if B[b][3] == 0:
            continue
        if prev is not None and (B[prev][2] > 0) != (B[b][2] > 0):
            rs = (prev + 0.5) + (b - prev) * B[prev][2] / (B[prev][2] - B[b][2])
            break
        prev = b
    gamma = 0.0 if rs != rs else sum(((b + 0.5) / rs) ** 2 * (B[b][0] - B[b][1]) for b in range(nb) if B[b][3] > 0 and b + 0.5 <= rmax)
    return dict(prof=prof, gsum=gsum, bins=bins, gamma=gamma, R_s=rs)


def _height(rho, fluid, z):
    """The softly weighted height of the droplet above the wall plane."""
    s = torch.sigmoid((rho[0] - rho[1]) / 0.05) * fluid
    return ((z - 0.5) * s).sum() / s.sum()


def exact(case, seed):
    kind = case["kind"]
    if kind == "sums":
        s = prepare(case, seed)
        n = s["n"] * (s["solid"] == 0)
        ex = _Exact(_solid(case), _params(case))
        c = ex.cons(n, 0)
        return c
    if kind == "sweep":
        out = dict(cons=[], rho=[], theta=[], theta_fit=[])
        for i, (e, p) in enumerate(_boxes(case)):
            box = dict(nx=e, ny=e, nz=e)
            ex = _Exact(_solid(box), p)
            n = ex.rest(*_sessile(box, seed + 31 * i))
            for _ in range(case["steps"]):
                n = ex.step(n)
            rho = ex.moments(n)[0]
            a = _droplet(rho[0] - rho[1], ex.solid, 5.0, 0.0)
            out["cons"].append(ex.cons(n, case["steps"]))
            out["rho"].append((rho[0], rho[1]))
            out["theta"].append(a["theta_deg"])
            out["theta_fit"].append(a["theta_fit_deg"])
        out["cons"] = torch.stack(out["cons"])
        return out
    ex = _Exact(_solid(case), _params(case))
    if kind == "step":
        n = ex.rest(*_step_fields(case, seed))
    else:
        n = ex.rest(*_sessile(case, seed, smooth=2.5 if kind in ("observe", "tension") else 0.0))
    if kind == "observe":
        rho = ex.moments(n)[0]
        phi = rho[0] - rho[1]
        zero = _droplet(phi, ex.solid, 5.0, 0.0)
        return dict(cons=ex.cons(n, 0), zero=zero, high=_droplet(phi, ex.solid, 5.0, 0.5 * zero["phi_max"]),
                    low=_droplet(phi, ex.solid, 5.0, 0.5 * zero["phi_min"]))
    if kind == "tension":
        for _ in range(20):
            n = ex.step(n)
        return _tension(ex, n, case)
    if kind == "adjoint":
        states = [n]
        for _ in range(case["steps"]):
            states.append(ex.step(states[-1]))
        fluid = ~ex.solid
        z = torch.arange(case["nz"], device=n.device, dtype=torch.float64)[:, None, None]
        last = states[-1].detach().requires_grad_()
        J = _height(ex.moments(last)[0], fluid, z)
        (lam,) = torch.autograd.grad(J, last)
        g = torch.zeros(2, dtype=torch.float64, device=n.device)
        for t in range(case["steps"] - 1, -1, -1):
            eta = ex.eta.clone().requires_grad_()
            x = states[t].detach().requires_grad_()
            lam, ge = torch.autograd.grad(ex.step(x, eta), (x, eta), lam)
            g = g + ge
        rho = ex.moments(states[-1])[0]
        return dict(J=float(J.detach()), g=g, rho_r=rho[0], rho_b=rho[1], cons=ex.cons(states[-1], case["steps"]))
    for _ in range(case["steps"]):
        n = ex.step(n)
    rho = ex.moments(n)[0]
    out = dict(rho_r=rho[0], rho_b=rho[1], cons=ex.cons(n, case["steps"]))
    if kind == "search":
        out.update(drop=_droplet(rho[0] - rho[1], ex.solid, 5.0, 0.0), u=ex.velocity(n))
    return out
