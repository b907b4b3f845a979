"""Workloads of the AICA pair-force library through its public entry points.

Each case is a call that a molecular-dynamics program makes on a mesh it
keeps: a velocity-Verlet step, the forces of a configuration, the gradient of
a loss on the forces, or the re-binning of molecules that have moved.  The
fluids are the library's own recipe: Lennard-Jones molecules on FCC sites at
reduced density 0.8 with Gaussian jitter, in jittered hexahedra, in Kuhn
tetrahedra, in a slab channel with posts and walls, or in a rotationally
periodic wedge.  The mesh of a case is fixed, as in a simulation; the seed
makes the molecules.

listed() and draw() give cases, prepare() and run() make and run one, work()
states what a pass cannot do without, and exact() gives the same results in
FP64 torch operations on a grid of cut-off sized cells.
"""
import functools
import math

import numpy as np
import torch

from paper_cs_0702131_gb300 import synth
from paper_cs_0702131_gb300.aica import LJForce, Mesh

DEV = "cuda"
A = (4.0 / 0.8) ** (1.0 / 3.0)          # FCC constant at reduced density 0.8
A_SC = (1.0 / 0.8) ** (1.0 / 3.0)       # simple cubic constant at the same density
BASIS = ((0.0, 0.0, 0.0), (0.5, 0.5, 0.0), (0.5, 0.0, 0.5), (0.0, 0.5, 0.5))
EPS = (1.0, 1.5)
SIGMA = (1.0, 0.88)
MASS = (1.0, 2.0)
SKIN = 1e-3
POSTS = ((0.25, 0.25), (0.75, 0.25), (0.25, 0.75), (0.75, 0.75))
POST_RADIUS = 5.0


def _case(name, kind, geom, fcc, grid, prec="fp32", species=1, rc=2.5, **more):
    c = dict(kind=kind, geom=geom, nx=fcc[0], ny=fcc[1], nz=fcc[2], gx=grid[0], gy=grid[1], gz=grid[2], prec=prec,
             species=species, rc=rc, shift=False, dt=0.002, move=0.0, deferred=False)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one step of a small simulation, thousands of them in a row: latency and launches
        _case("md_hex_2k", "md", "hex", (8, 8, 8), (6, 6, 6), shift=True, deferred=True),
        # one step of an ordinary simulation on a tetrahedral mesh
        _case("md_tet_256k", "md", "tet", (40, 40, 40), (24, 24, 24), deferred=True),
        # forces of a small configuration, checked at once (an interactive call)
        _case("forces_hex_4k", "forces", "hex", (10, 10, 10), (7, 7, 7)),
        # forces, energy, virial and pair counts of an ordinary configuration
        _case("forces_tet_256k", "forces", "tet", (40, 40, 40), (24, 24, 24)),
        # a nanochannel: open axis, walls of fixed molecules exactly on lattice planes, posts
        _case("forces_channel_1m", "forces", "channel", (144, 12, 144), (96, 10, 96)),
        # the largest: over a million molecules in half a million tetrahedra, longer cut-off
        _case("forces_tet_1m_rc3", "forces", "tet", (70, 70, 70), (44, 44, 44), rc=3.0),
        # reference-precision forces of a binary mixture
        _case("forces64_mix_64k", "forces", "hex", (16, 32, 32), (16, 16, 16), prec="fp64", species=2),
        # reference-precision forces on the tetrahedral mesh
        _case("forces64_tet_256k", "forces", "tet", (40, 40, 40), (24, 24, 24), prec="fp64"),
        # fitting potential parameters or positions: forces and their adjoint, two species
        _case("grad_mix_64k", "grad", "hex", (16, 32, 32), (16, 16, 16), species=2),
        # the same in reference precision, uneven box and mesh
        _case("grad64_tet_55k", "grad", "tet", (23, 25, 24), (14, 15, 13), prec="fp64"),
        # rotationally periodic domain (general referring transforms)
        _case("forces_wedge_129k", "forces", "wedge", (20, 100, 20), (32, 32, 12)),
        # molecules that moved half a diameter between two binnings (a long stride, a restart)
        _case("rebin_tet_256k", "bin", "tet", (40, 40, 40), (24, 24, 24), move=0.5),
    ]


def draw(rng):
    kind = rng.choice(["md", "md", "forces", "forces", "forces", "grad", "grad", "bin"])
    geom = rng.choice(["hex", "tet", "tet"])
    prec = rng.choice(["fp32", "fp32", "fp64"]) if kind != "bin" else "fp32"
    rc = rng.choice([2.5, 2.5, 3.0, round(rng.uniform(2.2, 3.2), 2)])
    species = rng.choice([1, 1, 2])
    top = {"fp32": 300000, "fp64": 120000}[prec]
    if kind == "forces" and rng.random() < 0.15:
        geom = "channel"
        k = int(round(math.exp(rng.uniform(math.log(24), math.log(110)))))
        h = rng.randint(8, 14)
        fcc = (k, h, max(24, k + rng.randint(-7, 7)))
        grid = (max(6, int(fcc[0] * A / 2.6)), rng.randint(7, 11), max(6, int(fcc[2] * A / 2.6)))
        return _case(None, kind, geom, fcc, grid, prec=prec if k < 60 else "fp32", rc=2.5)
    if kind == "forces" and rng.random() < 0.15:
        r0 = rng.randint(6, 20)
        fcc = (r0, r0 + rng.randint(12, 70), rng.randint(8, 20))
        grid = (max(3, int((fcc[1] - r0) / 2.6)), max(6, int(0.5 * math.pi * fcc[1] / 4.5)), max(4, int(fcc[2] * A_SC / 2.0)))
        return _case(None, kind, "wedge", fcc, grid, prec=prec, rc=2.5)
    n = math.exp(rng.uniform(math.log(700), math.log(top)))
    e = (n / 4.0) ** (1.0 / 3.0)
    fcc = tuple(max(5, int(round(e * rng.uniform(0.8, 1.25)))) for _ in range(3))
    w = rng.uniform(2.3, 3.4)                                   # width of a hexahedron
    grid = tuple(max(3, int(round(f * A / (w * rng.uniform(0.9, 1.1))))) for f in fcc)
    return _case(None, kind, geom, fcc, grid, prec=prec, species=species, rc=rc,
                 shift=kind in ("md", "forces") and rng.random() < 0.4, deferred=kind == "md" or rng.random() < 0.3,
                 move=rng.choice([0.01, 0.1, 0.5]) if kind == "bin" else 0.0)


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=3)
def _mesh(geom, nx, ny, nz, gx, gy, gz):
    """The case's mesh, box and (wedge) transforms: fixed, as a program's mesh file is."""
    if geom == "channel":
        Lx, Lz = nx * A, nz * A
        lo, hi = (0.0, -1.25 * A, 0.0), (Lx, (ny + 0.75) * A, Lz)
        cx, cz = np.meshgrid((np.arange(gx) + 0.5) * Lx / gx, (np.arange(gz) + 0.5) * Lz / gz, indexing="ij")
        post = np.zeros_like(cx, dtype=bool)
        for fx, fz in POSTS:
            post |= (cx - fx * Lx) ** 2 + (cz - fz * Lz) ** 2 < POST_RADIUS ** 2
        removed = np.broadcast_to(post[:, None, :], (gx, gy, gz)).reshape(-1)
        mesh = synth.hex_mesh((gx, gy, gz), lo, hi, 0.15, np.random.default_rng(5), keep=~removed)
        return mesh, dict(L=np.array([Lx, hi[1] - lo[1], Lz]), periodic=np.array([1, 0, 1], np.int32)), post
    if geom == "wedge":
        c = synth.wedge(0, r0=float(nx), r1=float(ny), nz_sc=nz, nr=gx, ntheta=gy, nz=gz)
        return c["mesh"], c["box"], c["transforms"]
    L = np.array([nx, ny, nz]) * A
    mesh = synth.hex_mesh((gx, gy, gz), (0, 0, 0), L, 0.15, np.random.default_rng(5), tets=geom == "tet")
    return mesh, dict(L=L, periodic=np.array([1, 1, 1], np.int32)), None


def _geom(c):
    return tuple(c[k] for k in ("geom", "nx", "ny", "nz", "gx", "gy", "gz"))


def _sites(nx, ny, nz, y0=0):
    i, j, k = torch.meshgrid(torch.arange(nx, device=DEV), torch.arange(y0, y0 + ny, device=DEV),
                             torch.arange(nz, device=DEV), indexing="ij")
    cells = torch.stack([i, j, k], -1).reshape(-1, 1, 3).double()
    return ((cells + torch.tensor(BASIS, dtype=torch.float64, device=DEV)) * A).reshape(-1, 3)


def _wrap(x, L, periodic):
    for d in range(3):
        if periodic[d]:
            x[:, d] -= L[d] * torch.floor(x[:, d] / L[d])
            x[:, d] = torch.where(x[:, d] >= L[d], torch.zeros_like(x[:, d]), x[:, d])
    return x


def _inputs(c, seed):
    """Molecules of the case: positions, species and what the kind needs besides."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)

    def normal(*shape):
        return torch.randn(*shape, generator=g, dtype=torch.float64, device=DEV)

    _, box, more = _mesh(*_geom(c))
    L, per = [float(v) for v in box["L"]], [int(v) for v in box["periodic"]]
    if c["geom"] == "channel":
        pos = _sites(c["nx"], c["ny"] + 2, c["nz"], -1)
        fluid = ((pos[:, 1] > -1e-9) & (pos[:, 1] < c["ny"] * A - 1e-9))[:, None]
        post = torch.tensor(more, device=DEV)
        gap = torch.where(fluid[:, 0], 0.2, 1e-7)       # no molecule inside a removed hexahedron, nor on its faces
        keep = torch.ones(pos.shape[0], dtype=torch.bool, device=DEV)
        for ex in (-1, 1):
            for ez in (-1, 1):
                ix = torch.floor((pos[:, 0] + ex * gap) * (c["gx"] / L[0])).long() % c["gx"]
                iz = torch.floor((pos[:, 2] + ez * gap) * (c["gz"] / L[2])).long() % c["gz"]
                keep &= ~post[ix, iz]
        pos, fluid = pos[keep], fluid[keep]
        pos = _wrap(torch.where(fluid, pos + 0.05 * normal(*pos.shape).clamp(-3.9, 3.9), pos), L, per).contiguous()
    elif c["geom"] == "wedge":
        r0, r1, H = float(c["nx"]), float(c["ny"]), c["nz"] * A_SC
        n1 = int(math.ceil(r1 / A_SC)) + 1
        ax = [(torch.arange(m, device=DEV).double() + 0.5) * A_SC for m in (n1, n1, c["nz"])]
        pos = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)
        rad = torch.hypot(pos[:, 0], pos[:, 1])
        pos = pos[(rad > r0 + 0.2) & (rad < r1 * math.cos(0.25 * math.pi / c["gy"]) - 0.2)]
        pos = pos + 0.05 * normal(*pos.shape).clamp(-3.5, 3.5)
        pos[:, 2].clamp_(1e-6, H - 1e-6)
        pos = pos[(pos[:, 0] > 1e-6) & (pos[:, 1] > 1e-6)].contiguous()
    else:
        pos = _sites(c["nx"], c["ny"], c["nz"])
        pos = _wrap(pos + 0.05 * normal(*pos.shape), L, per)
    n = pos.shape[0]
    sp = torch.zeros(n, dtype=torch.int32, device=DEV)
    if c["species"] == 2:
        sp[torch.randperm(n, generator=g, device=DEV)[: n // 2]] = 1
    s = dict(pos=pos, species=sp, eps=EPS[: c["species"]], sigma=SIGMA[: c["species"]])
    if c["kind"] == "md":
        m = torch.tensor(MASS, dtype=torch.float64, device=DEV)[sp.long()][:, None]
        v = normal(n, 3) / m.sqrt()
        s["vel"] = v - (m * v).sum(0) / m.sum()
    elif c["kind"] == "grad":
        s["grad"] = normal(n, 3).to(torch.float32 if c["prec"] == "fp32" else torch.float64)
    elif c["kind"] == "bin":
        v = normal(n, 3)
        s["moved"] = _wrap(pos + c["move"] * v / v.norm(dim=1, keepdim=True), L, per)
    return s


def prepare(case, seed):
    c = case
    mesh, box, more = _mesh(*_geom(c))
    s = _inputs(c, seed)
    m = Mesh(mesh, box)
    if c["geom"] == "wedge":
        m.set_transforms(more)
    m.build_lists(c["rc"], SKIN)
    s.update(case=c, mesh=m, n=s["pos"].shape[0])
    if c["kind"] == "md":
        m.bin(s["pos"], s["species"], outputs=False)
        s["force"] = m.forces(s["eps"], s["sigma"], c["prec"], shift=c["shift"])[0]
        s["ev"] = torch.empty(7, dtype=torch.float64, device=DEV)
        s["kin"] = torch.empty(4, dtype=torch.float64, device=DEV)
        s["mass"] = MASS[: c["species"]]
    elif c["kind"] == "grad":
        s["eps_t"] = torch.tensor(s["eps"], dtype=torch.float64, requires_grad=True)
        s["sigma_t"] = torch.tensor(s["sigma"], dtype=torch.float64, requires_grad=True)
        s["pos"].requires_grad_(True)
    m.set_deferred(c["deferred"])
    return s


def run(s):
    c, m = s["case"], s["mesh"]
    if c["kind"] == "md":
        m.verlet_step(s["eps"], s["sigma"], s["mass"], c["dt"], s["pos"], s["vel"], s["species"], s["force"],
                      prec=c["prec"], ev=s["ev"], kin=s["kin"], shift=c["shift"])
        return {k: s[k] for k in ("pos", "vel", "force", "ev", "kin")}
    if c["kind"] == "grad":
        F = LJForce.apply(s["pos"], s["eps_t"], s["sigma_t"], m, s["species"], c["prec"])
        gp, ge, gs = torch.autograd.grad(F, (s["pos"], s["eps_t"], s["sigma_t"]), s["grad"])
        return dict(force=F.detach(), grad_pos=gp, grad_eps=ge, grad_sigma=gs)
    if c["kind"] == "bin":
        a = m.bin(s["pos"], s["species"])
        b = m.bin(s["moved"], s["species"])
        return dict(first=list(a), second=list(b))
    m.bin(s["pos"], s["species"], outputs=False)
    F, ev, counts = m.forces(s["eps"], s["sigma"], c["prec"], shift=c["shift"])
    return dict(force=F, ev=ev, counts=counts)


def work(case):
    c = case
    if c["geom"] == "wedge":
        n = 0.8 * 0.25 * math.pi * (c["ny"] ** 2 - c["nx"] ** 2) * c["nz"] * A_SC
    elif c["geom"] == "channel":
        n = 4.0 * c["nx"] * (c["ny"] + 2) * c["nz"] - 4 * math.pi * POST_RADIUS ** 2 * (c["ny"] + 2) * A * 0.8
    else:
        n = 4.0 * c["nx"] * c["ny"] * c["nz"]
    cells = c["gx"] * c["gy"] * c["gz"] * (6 if c["geom"] == "tet" else 1)
    real = 8 if c["prec"] == "fp64" else 4
    pairs = 0.5 * n * 0.8 * 4.0 / 3.0 * math.pi * c["rc"] ** 3     # within the cut-off, each once
    if c["kind"] == "bin":
        return {"bytes": 2 * (n * (24 + 4 + 8) + 4 * cells), "flops": 0}
    if c["kind"] == "md":       # positions, velocities and forces in and out, species in
        return {"bytes": n * (2 * 24 + 2 * 24 + 6 * real + 4), "flops": 32 * pairs}
    if c["kind"] == "grad":     # positions, species, dL/dF in; forces and dL/dx out
        return {"bytes": n * (24 + 4 + 3 * real + 3 * real + 24), "flops": (32 + 50) * pairs}
    return {"bytes": n * (24 + 4 + 3 * real), "flops": 32 * pairs}


# ------------------------------------------------------------------ exact values (FP64 torch)
def _images(c, x):
    """x and its periodic images within the cut-off of the domain, with their sources."""
    _, box, more = _mesh(*_geom(c))
    reach = c["rc"] + 1e-6
    src = torch.arange(x.shape[0], device=DEV)
    if c["geom"] == "wedge":
        H = c["nz"] * A_SC
        q, s = [x], [src]
        for a in (0, 1, -1):
            y = x if a == 0 else torch.stack([-x[:, 1], x[:, 0], x[:, 2]], 1) if a == 1 else \
                torch.stack([x[:, 1], -x[:, 0], x[:, 2]], 1)
            for b in (0, 1, -1):
                if a or b:
                    z = y + torch.tensor([0.0, 0.0, b * H], dtype=torch.float64, device=DEV)
                    keep = (z[:, 0] > -reach) & (z[:, 1] > -reach) & (z[:, 2] > -reach) & (z[:, 2] < H + reach)
                    q.append(z[keep])
                    s.append(src[keep])
        return torch.cat(q), torch.cat(s)
    q, s = x, src
    for d in range(3):
        if box["periodic"][d]:
            L = float(box["L"][d])
            low, high = q[:, d] < reach, q[:, d] >= L - reach
            up, down = q[low].clone(), q[high].clone()
            up[:, d] += L
            down[:, d] -= L
            q, s = torch.cat([q, up, down]), torch.cat([s, s[low], s[high]])
    return q, s


def _neighbours(c, x):
    """Blocks (rows i, sources [i, m], separations x_i - q [i, m, 3], within the cut-off [i, m])."""
    q, src = _images(c, x)
    w = c["rc"] * (1 + 1e-9)
    lo = q.min(0).values - 1e-9
    G = [int(v) + 3 for v in ((q.max(0).values - lo) / w).tolist()]

    def cell(p):
        k = ((p - lo) / w).long() + 1
        return (k[:, 0] * G[1] + k[:, 1]) * G[2] + k[:, 2]

    cq = cell(q)
    order = torch.argsort(cq)
    off = torch.zeros(G[0] * G[1] * G[2] + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(cq, minlength=off.shape[0] - 1), 0)
    q, src, self_at = q[order], src[order], torch.empty_like(order)
    self_at[order] = torch.arange(order.shape[0], device=DEV)
    home = cell(x)
    step = 1 << 15
    for i0 in range(0, x.shape[0], step):
        rows = torch.arange(i0, min(i0 + step, x.shape[0]), device=DEV)
        for dx in (-1, 0, 1):
            for dy in (-1, 0, 1):
                k = home[rows] + (dx * G[1] + dy) * G[2]
                a, b = off[k - 1], off[k + 2]
                m = int((b - a).max())
                if m == 0:
                    continue
                j = a[:, None] + torch.arange(m, device=DEV)
                ok = (j < b[:, None]) & (j != self_at[rows][:, None])
                j = j.clamp(max=q.shape[0] - 1)
                r = x[rows][:, None, :] - q[j]
                ok &= (r * r).sum(-1) < c["rc"] ** 2
                ii, mm = ok.nonzero(as_tuple=True)
                yield rows[ii], src[j[ii, mm]], r[ii, mm]


def _lj(c, x, sp, v=None):
    """F, (U, W), and with v = dL/dF the position and species gradients."""
    eps = torch.tensor(EPS[: c["species"]], dtype=torch.float64, device=DEV)
    sig = torch.tensor(SIGMA[: c["species"]], dtype=torch.float64, device=DEV)
    F, ev = torch.zeros_like(x), torch.zeros(7, dtype=torch.float64, device=DEV)
    gp, ge, gs = torch.zeros_like(x), torch.zeros_like(eps), torch.zeros_like(sig)
    sp = sp.long()
    for i, j, r in _neighbours(c, x):
        a, b = sp[i], sp[j]
        e, s = (eps[a] * eps[b]).sqrt(), 0.5 * (sig[a] + sig[b])
        r2 = (r * r).sum(-1)
        s6 = (s * s / r2) ** 3
        f = 24 * e * s6 * (2 * s6 - 1) / r2
        fv = f[:, None] * r
        F.index_add_(0, i, fv)
        u = 4 * e * s6 * (s6 - 1)
        if c["shift"]:
            sc = (s * s / c["rc"] ** 2) ** 3
            u = u - 4 * e * sc * (sc - 1)
        ev[0] += 0.5 * u.sum()
        for k, (p, q) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            ev[1 + k] += 0.5 * (r[:, p] * fv[:, q]).sum()
        if v is not None:
            w = v[i] - v[j]
            rw = (r * w).sum(-1)
            gp.index_add_(0, i, f[:, None] * w + (2 * 24 * e * s6 * (4 - 14 * s6) / (r2 * r2) * rw)[:, None] * r)
            de, dsg = 0.5 * f * rw / e, 0.5 * 24 * e * s6 * (24 * s6 - 6) / r2 * rw / s
            for p, q in ((a, b), (b, a)):
                ge.index_add_(0, p, de * 0.5 * e / eps[p])
                gs.index_add_(0, p, 0.5 * dsg)
    return F, ev, gp, ge, gs


def exact(case, seed):
    c = case
    if c["kind"] == "bin":
        return None
    s = _inputs(c, seed)
    x, sp = s["pos"].detach().clone(), s["species"]
    _, box, _ = _mesh(*_geom(c))
    if c["kind"] == "md":
        m = torch.tensor(MASS, dtype=torch.float64, device=DEV)[sp.long()][:, None]
        v = s["vel"] + 0.5 * c["dt"] * _lj(c, x, sp)[0] / m
        x = x + c["dt"] * v
        F, ev = _lj(c, _wrap(x.clone(), [float(t) for t in box["L"]], box["periodic"]), sp)[:2]
        v = v + 0.5 * c["dt"] * F / m
        kin = torch.cat([(0.5 * m * v * v).sum().reshape(1), (m * v).sum(0)])
        return dict(pos=x, vel=v, force=F, ev=ev, kin=kin)
    if c["kind"] == "grad":
        F, _, gp, ge, gs = _lj(c, x, sp, s["grad"].double())
        return dict(force=F, grad_pos=gp, grad_eps=ge, grad_sigma=gs)
    F, ev = _lj(c, x, sp)[:2]
    return dict(force=F, ev=ev, counts=None)
