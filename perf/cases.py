"""What a user of the GFM pressure solver has it do, as measurable cases.

A case is one call (or the short sequence of calls) that a free-surface flow
program makes through the public entry points: a pressure solve of a wave
tank or of a green-water box (assembly included, because alpha and the
predicted flux are new at every call), a batch of tanks, the pressure part of
a time step, a differentiable solve with its backward pass, and the steps
around the solve (gradient and velocity, non-orthogonal correction,
isoAdvector step, the solve of a caller's CSR matrix).

Meshes are hexahedral with walls all round, as in the repository's workloads:
uniform (tanks, boxes), smoothly distorted (non-orthogonal) or graded, in the
caller's natural cell order or in a random one.  The handle is made once per
mesh and kept, as a program does; alpha, fluxes and p_d come new.

Solves are asked for a true relative residual of 1e-12 (1e-11 on the
box), tight enough that two correct solvers agree in p_d to nine digits.
They return p_d.  The corrected flux and quantities derived from it are small
differences of large terms there (phi* and gamma grad p_d against the jump),
so they are measured on a given p_d, in the cases of the steps around the
solve.
"""
import math

import numpy as np
import torch

import paper_1804_01130_gb300 as gfm

RHO_W, RHO_A, GRAV = 1000.0, 1.0, (0.0, -9.81, 0.0)
DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # the smallest pressure solve: 64 x 32 cells in plain FP64, a coarse
        # study or one tank of a teaching example; latency is all there is
        dict(name="tank_64x32_fp64", kind="solve", nx=64, ny=32, nz=1, lx=2.0, ly=1.0, ka=0.12, waves=2, mode="fp64",
             rtol=1e-12, permute=False, renumber=1),
        # the 2D progressive-wave tank at the resolution of the benchmark
        dict(name="tank_1024x512_mixed", kind="solve", nx=1024, ny=512, nz=1, lx=16.0, ly=4.0, ka=0.1, waves=4,
             mode="mixed", rtol=1e-12, permute=False, renumber=1),
        # the same problem from a host program's buffers, an odd size: copies
        # in, assembly, solve and copy out in one call
        dict(name="tank_host_601x203", kind="host", nx=601, ny=203, nz=1, lx=16.0, ly=4.0, ka=0.08, waves=3,
             mode="mixed", rtol=1e-12, permute=False, renumber=1),
        # the 3D green-water box, 4.2M cells in a random caller order: the
        # largest mesh, streamed from HBM
        dict(name="box_256x128x128_mixed", kind="solve", nx=256, ny=128, nz=128, lx=4.0, ly=2.0, ka=0.0, waves=0,
             mode="mixed", rtol=1e-11, permute=True, renumber=1),
        # many tanks of uneven size in one launch (a design-space study)
        dict(name="batch_64", kind="batch", tanks=64, nx_lo=128, nx_hi=1024, ny_lo=64, ny_hi=256, rtol=1e-12,
             renumber=1),
        # the pressure part of one time step: 6 outer iterations x 2
        # correctors, warm-started
        dict(name="step_1024x512", kind="step", nx=1024, ny=512, nz=1, lx=16.0, ly=4.0, ka=0.1, waves=4, solves=12,
             mode="mixed", rtol=1e-12, permute=False, renumber=1),
        # a differentiable solve and its backward pass (adjoint) in FP64
        dict(name="adjoint_256x128", kind="adjoint", nx=256, ny=128, nz=1, lx=4.0, ly=2.0, ka=0.1, waves=2,
             mode="fp64", rtol=1e-12, permute=False, renumber=1),
        # a solver plugged into a host program that owns the device memory
        dict(name="csr_300x200", kind="csr", nx=300, ny=200, nz=1, lx=6.0, ly=4.0, ka=0.1, waves=2, rtol=1e-12),
        # assembly of the box with the assembled system read back (a program
        # with its own solver, or its own diagnostics)
        dict(name="assemble_256x128x128", kind="assemble", nx=256, ny=128, nz=128, lx=4.0, ly=2.0, ka=0.0, waves=0,
             permute=True, renumber=1),
        # the momentum equation's pressure gradient and the reconstructed
        # velocity on a ragged 3D mesh
        dict(name="gradient_201x101x99", kind="gradient", nx=201, ny=101, nz=99, lx=4.0, ly=2.0, ka=0.0, waves=0,
             permute=True, renumber=1),
        # one deferred non-orthogonal correction on a distorted mesh
        dict(name="nonorth_769x513", kind="nonorth", nx=769, ny=513, eps=0.04, renumber=1),
        # one isoAdvector step on a graded 3D mesh
        dict(name="iso_128x96x64", kind="iso", nx=128, ny=96, nz=64, renumber=1),
    ]


# ---------------------------------------------------------------------------
# the ranges that the listed cases stand for
# ---------------------------------------------------------------------------
def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _tank(rng, cells_lo, cells_hi):
    """A tank's sizes: cells within the range, height/width of the cells
    between 1/4 and 4, as in the batch's tanks."""
    while True:
        nx, ny = _log_int(rng, 24, 2048), _log_int(rng, 12, 768)
        if cells_lo <= nx * ny <= cells_hi:
            break
    ly = rng.uniform(1.0, 4.0)
    lx = ly * nx / ny * math.exp(rng.uniform(-math.log(4.0), math.log(4.0)))
    return dict(nx=nx, ny=ny, nz=1, lx=round(lx, 3), ly=round(ly, 3), ka=round(rng.uniform(0.02, 0.15), 3),
                waves=rng.randint(1, 6))


def _box(rng, cells_lo, cells_hi):
    while True:
        nx, ny, nz = _log_int(rng, 16, 256), _log_int(rng, 12, 128), _log_int(rng, 12, 128)
        if cells_lo <= nx * ny * nz <= cells_hi:
            break
    return dict(nx=nx, ny=ny, nz=nz, lx=4.0, ly=2.0, ka=0.0, waves=0)


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "host", "batch", "step", "adjoint", "csr", "assemble", "gradient",
                       "nonorth", "iso"])
    ren = rng.choice([0, 1, 1, 1, 2])
    if kind in ("solve", "host"):
        three = rng.random() < 0.4
        mode = "mixed" if kind == "host" else rng.choice(["mixed", "mixed", "fp64"])
        top = 4_194_304 if mode == "mixed" else 600_000
        c = _box(rng, 4000, top) if three else _tank(rng, 800, min(top, 1_000_000))
        perm = rng.random() < 0.3
        if perm:
            ren = rng.choice([1, 1, 2])
        return dict(kind=kind, **c, mode=mode, rtol=1e-11 if three else 1e-12, permute=perm, renumber=ren)
    if kind == "batch":
        lo = _log_int(rng, 24, 160)
        return dict(kind="batch", tanks=_log_int(rng, 2, 64), nx_lo=lo, nx_hi=lo * rng.randint(2, 6), ny_lo=lo // 2,
                    ny_hi=min(256, lo * 2), rtol=1e-12, renumber=1)
    if kind == "step":
        return dict(kind="step", **_tank(rng, 2000, 524_288), solves=rng.choice([4, 6, 12]), mode="mixed", rtol=1e-12,
                    permute=False, renumber=ren)
    if kind == "adjoint":
        return dict(kind="adjoint", **_tank(rng, 800, 32_768), mode="fp64", rtol=1e-12, permute=False, renumber=ren)
    if kind == "csr":
        return dict(kind="csr", **_tank(rng, 800, 120_000), rtol=1e-12)
    if kind in ("assemble", "gradient"):
        c = _box(rng, 4000, 4_194_304) if rng.random() < 0.6 else _tank(rng, 800, 1_000_000)
        return dict(kind=kind, **c, permute=rng.random() < 0.5, renumber=ren)
    if kind == "nonorth":
        while True:
            nx, ny = _log_int(rng, 24, 1024), _log_int(rng, 16, 768)
            if nx * ny <= 500_000:
                break
        return dict(kind="nonorth", nx=nx, ny=ny, eps=round(rng.uniform(0.01, 0.05), 3), renumber=ren)
    while True:
        nx, ny, nz = _log_int(rng, 12, 160), _log_int(rng, 12, 128), _log_int(rng, 8, 96)
        if nx * ny * nz <= 786_432:
            break
    return dict(kind="iso", nx=nx, ny=ny, nz=nz, renumber=ren)


# ---------------------------------------------------------------------------
# meshes and fields, made on the GPU from the seed
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _cells(nx, ny, nz):
    idx = torch.arange(nx * ny * nz, device=DEV)
    return idx, idx % nx, (idx // nx) % ny, idx // (nx * ny)


def _faces(nx, ny, nz):
    """owner, neighbour and axis of every internal face, sorted by (owner, neighbour)."""
    idx, i, j, k = _cells(nx, ny, nz)
    has = torch.stack([i < nx - 1, j < ny - 1, k < nz - 1], dim=1)
    step = torch.tensor([1, nx, nx * ny], device=DEV)
    o = idx[:, None].expand(-1, 3)[has]
    ax = torch.arange(3, device=DEV)[None].expand(idx.numel(), 3)[has]
    return o, o + step[ax], ax


def _uniform(nx, ny, nz, lx, ly):
    """A uniform hex mesh lx x ly, one cell of width dx deep in 2D, lz = lx/2 in 3D."""
    dx, dy = lx / nx, ly / ny
    dz = dx if nz == 1 else 0.5 * lx / nz
    _, i, j, k = _cells(nx, ny, nz)
    C = torch.stack([(i + 0.5) * dx, (j + 0.5) * dy, (k + 0.5) * dz]).to(F64)
    o, v, ax = _faces(nx, ny, nz)
    h = torch.tensor([dx, dy, dz], device=DEV, dtype=F64)
    area = torch.tensor([dy * dz, dx * dz, dx * dy], device=DEV, dtype=F64)
    S = torch.zeros((3, o.numel()), device=DEV, dtype=F64)
    S.scatter_(0, ax[None], area[ax][None])
    xf = C[:, o]
    xf.scatter_add_(0, ax[None], (0.5 * h)[ax][None])
    V = torch.full((nx * ny * nz,), dx * dy * dz, device=DEV, dtype=F64)
    return dict(n=nx * ny * nz, F=o.numel(), owner=o, neighbour=v, Sf=S, C=C, V=V, xf=xf, h=(dx, dy, dz),
                dims=(nx, ny, nz))


def _permute(m, g, fields=()):
    """The mesh in a random cell order; face fields (oriented) follow their faces."""
    n = m["n"]
    perm = torch.randperm(n, device=DEV, generator=g)
    o, v = perm[m["owner"]], perm[m["neighbour"]]
    flip = o > v
    o, v = torch.where(flip, v, o), torch.where(flip, o, v)
    order = torch.argsort(o * n + v)
    sgn = torch.where(flip, -1.0, 1.0).to(F64)
    back = torch.empty_like(perm)
    back[perm] = torch.arange(n, device=DEV)
    out = dict(m, owner=o[order], neighbour=v[order], Sf=(m["Sf"] * sgn)[:, order].contiguous(),
               C=m["C"][:, back].contiguous(), V=m["V"][back].contiguous(), xf=m["xf"][:, order].contiguous(),
               perm=perm, order=order, sgn=sgn)
    return out, [(f * sgn)[order].contiguous() for f in fields]


def _eta(x, lx, ly, ka, waves):
    """Second-order Stokes surface elevation over a depth of ly/2."""
    k = 2.0 * math.pi * waves / lx
    depth = 0.5 * ly
    a, kd = ka / k, min(k * depth, 30.0)
    a = min(a, 0.3 * depth)
    a2 = (k * a * a / 4.0) * math.cosh(kd) * (2.0 + math.cosh(2.0 * kd)) / math.sinh(kd) ** 3
    return depth + a * torch.cos(k * x) + a2 * torch.cos(2.0 * k * x)


def _alpha(m, c, g):
    """Volume fraction: under a wave in 2D; a layer with bumps, a dam-break column and spheres in 3D."""
    C, (dx, dy, dz) = m["C"], m["h"]
    lx, ly = c["lx"], c["ly"]
    phase = lx * torch.rand(1, device=DEV, generator=g, dtype=F64)
    a = torch.zeros(m["n"], device=DEV, dtype=F64)
    if c["nz"] == 1:
        for q in range(8):
            x = C[0] + ((q + 0.5) / 8 - 0.5) * dx
            a += ((_eta(x + phase, lx, ly, c["ka"], c["waves"]) - (C[1] - 0.5 * dy)) / dy).clamp(0.0, 1.0)
        return a / 8
    r = torch.rand((8, 4), device=DEV, generator=g, dtype=F64)
    amp, sig, cx, cz = 0.05 + 0.25 * r[:, 0], 0.1 + 0.3 * r[:, 1], lx * r[:, 2], 0.5 * lx * r[:, 3]
    s = torch.rand((6, 4), device=DEV, generator=g, dtype=F64)
    sx, sy, sz, sr = 0.3 + (lx - 0.6) * s[:, 0], 1.2 + 0.55 * s[:, 1], 0.3 + (0.5 * lx - 0.6) * s[:, 2], 0.05 + 0.15 * s[:, 3]
    for q in range(27):
        x = C[0] + ((q % 3) - 1) * dx / 3
        y = C[1] + ((q // 3 % 3) - 1) * dy / 3
        z = C[2] + (q // 9 - 1) * dz / 3
        top = torch.full_like(x, 0.6)
        for b in range(8):
            top += amp[b] * torch.exp(-((x - cx[b]) ** 2 + (z - cz[b]) ** 2) / (2.0 * sig[b] ** 2))
        w = (y < top) | ((x < 1.0) & (y < 1.4))
        for b in range(6):
            w |= (x - sx[b]) ** 2 + (y - sy[b]) ** 2 + (z - sz[b]) ** 2 < sr[b] ** 2
        a += w
    return a / 27


def _flux(m, g, amp=0.1):
    """A predicted face flux S_f . u(x_f), u a sum of 8 smooth modes, not divergence-free."""
    two = m["dims"][2] == 1
    kmax = 2.0 * math.pi / (4.0 * (min(m["h"][:2]) if two else min(m["h"])))
    xf = m["xf"]
    r = torch.rand((8, 8), device=DEV, generator=g, dtype=F64)
    out = torch.zeros(m["F"], device=DEV, dtype=F64)
    for q in range(8):
        a = amp * (2.0 * r[q, 0:3] - 1.0)
        d = 2.0 * r[q, 3:6] - 1.0
        if two:
            a[2] = 0.0
            d[2] = 0.0
        kv = d / d.norm().clamp_min(1e-12) * (kmax * r[q, 6])
        arg = kv[0] * xf[0] + kv[1] * xf[1] + kv[2] * xf[2] + 2.0 * math.pi * r[q, 7]
        out += (a @ m["Sf"]) * (torch.sin(arg) if q % 2 == 0 else torch.cos(arg))
    return out


def _wavy(nx, ny, eps):
    """Nodes of a smoothly distorted quadrilateral mesh of 2 x 1, extruded one cell deep."""
    lx, ly = 2.0, 1.0
    y, x = torch.meshgrid(torch.linspace(0, ly, ny + 1, device=DEV, dtype=F64),
                          torch.linspace(0, lx, nx + 1, device=DEV, dtype=F64), indexing="ij")
    X = x + eps * lx * torch.sin(math.pi * x / lx) * torch.sin(2 * math.pi * y / ly)
    Y = y + eps * ly * torch.sin(2 * math.pi * x / lx) * torch.sin(math.pi * y / ly)
    dz = lx / nx
    vx = torch.stack([X[:-1, :-1], X[:-1, 1:], X[1:, 1:], X[1:, :-1]], -1).reshape(-1, 4)
    vy = torch.stack([Y[:-1, :-1], Y[:-1, 1:], Y[1:, 1:], Y[1:, :-1]], -1).reshape(-1, 4)
    x1, y1 = vx.roll(-1, 1), vy.roll(-1, 1)
    cr = vx * y1 - x1 * vy
    ar = 0.5 * cr.sum(1)
    C = torch.stack([((vx + x1) * cr).sum(1) / (6 * ar), ((vy + y1) * cr).sum(1) / (6 * ar), torch.full_like(ar, dz / 2)])
    o, v, ax = _faces(nx, ny, 1)
    i, j = o % nx, o // nx
    # the edge of a face: between (i, j) and its neighbour in +x or in +y
    bx0, by0 = torch.where(ax == 0, i + 1, i + 1), torch.where(ax == 0, j, j + 1)
    bx1, by1 = torch.where(ax == 0, i + 1, i), j + 1
    ex0, ey0, ex1, ey1 = X[by0, bx0], Y[by0, bx0], X[by1, bx1], Y[by1, bx1]
    S = torch.stack([(ey1 - ey0) * dz, -(ex1 - ex0) * dz, torch.zeros_like(ex0)])
    xf = torch.stack([0.5 * (ex0 + ex1), 0.5 * (ey0 + ey1), torch.full_like(ex0, dz / 2)])
    return dict(n=nx * ny, F=o.numel(), owner=o, neighbour=v, Sf=S.contiguous(), C=C.contiguous(), V=ar * dz, xf=xf,
                h=(lx / nx, ly / ny, dz), dims=(nx, ny, 1))


def _graded(nx, ny, nz, g):
    """A tensor-product mesh of uneven cells with its face polygons (four corners a face)."""
    nodes = []
    for m, length in ((nx, 4.0), (ny, 2.0), (nz, 2.0)):
        w = 0.6 + 0.8 * torch.rand(m, device=DEV, generator=g, dtype=F64)
        nodes.append(torch.cat([torch.zeros(1, device=DEV, dtype=F64), torch.cumsum(w, 0)]) * (length / w.sum()))
    _, i, j, k = _cells(nx, ny, nz)
    ijk = torch.stack([i, j, k])
    lo = torch.stack([nodes[a][ijk[a]] for a in range(3)])
    hi = torch.stack([nodes[a][ijk[a] + 1] for a in range(3)])
    C, d = 0.5 * (lo + hi), hi - lo
    o, v, ax = _faces(nx, ny, nz)
    area = torch.stack([d[1] * d[2], d[0] * d[2], d[0] * d[1]])
    S = torch.zeros((3, o.numel()), device=DEV, dtype=F64)
    S.scatter_(0, ax[None], area[ax, o][None])
    flo, fhi = lo[:, o].clone(), hi[:, o]
    flo.scatter_(0, ax[None], torch.gather(fhi, 0, ax[None]))  # both corners on the face's plane
    xf = 0.5 * (flo + fhi)
    u, w = torch.where(ax == 0, 1, 0), torch.where(ax == 2, 1, 2)
    corners = []
    for cu, cw in ((0, 0), (1, 0), (1, 1), (0, 1)):
        p = flo.clone()
        if cu:
            p.scatter_(0, u[None], torch.gather(fhi, 0, u[None]))
        if cw:
            p.scatter_(0, w[None], torch.gather(fhi, 0, w[None]))
        corners.append(p)
    xyz = torch.stack(corners, dim=2).reshape(3, -1).contiguous()
    ptr = torch.arange(0, 4 * o.numel() + 1, 4, device=DEV, dtype=torch.int32)
    return dict(n=nx * ny * nz, F=o.numel(), owner=o, neighbour=v, Sf=S, C=C, V=d.prod(0), xf=xf, fv_ptr=ptr, fv_xyz=xyz,
                h=tuple(float(t.min()) for t in d), dims=(nx, ny, nz))


def _problem(c, seed):
    """Mesh, alpha and predicted flux of a tank or box, in structured and in caller order."""
    g = _gen(seed)
    m = _uniform(c["nx"], c["ny"], c["nz"], c["lx"], c["ly"])
    alpha, phi = _alpha(m, c, g), _flux(m, g)
    ref = (c["ny"] - 1) * c["nx"]  # the top-left cell
    u, a_u, f_u = m, alpha, phi
    if c.get("permute"):
        m, (phi,) = _permute(u, g, (phi,))
        alpha = torch.empty_like(a_u)
        alpha[m["perm"]] = a_u
        ref_c = int(m["perm"][ref])
    else:
        ref_c = ref
    phys = dict(rho_w=RHO_W, rho_a=RHO_A, g=GRAV, ref_cell=ref_c, ref_value=0.0)
    return dict(m=m, alpha=alpha.contiguous(), phi=phi.contiguous(), phys=phys, u=u, a_u=a_u, f_u=f_u, ref=ref, g=g)


def _handle(m, c):
    return gfm.GFM(m["owner"], m["neighbour"], m["Sf"], m["C"], renumber=c["renumber"])


def _correctors(q, k):
    """Predicted fluxes of a time step's correctors: changes that shrink by 0.6 per corrector."""
    out = [q["phi"]]
    for j in range(1, k):
        out.append(out[-1] + 0.6 ** j * _flux(q["m"], q["g"]))
    return torch.stack(out)


def _pressure_like(m, q):
    """A p_d of the size of a solution: the hydrostatic jump across the surface plus a smooth field."""
    C, g = m["C"], q["g"]
    r = torch.rand(4, device=DEV, generator=g, dtype=F64)
    smooth = 200.0 * torch.sin(2.0 * r[0] * C[0] + 6.0 * r[1]) * torch.cos(3.0 * r[2] * C[1] + r[3])
    return (q["alpha"] * (19620.0 + smooth) + (1.0 - q["alpha"]) * 0.001 * smooth).contiguous()


def _tank_case(c, t, seed):
    """Tank t of a batch: the sizes belong to the case, the fields to the seed."""
    r = np.random.default_rng(4000 + t)
    return dict(nx=int(r.integers(c["nx_lo"], c["nx_hi"] + 1)), ny=int(r.integers(c["ny_lo"], c["ny_hi"] + 1)), nz=1,
                lx=16.0, ly=4.0, ka=float(r.uniform(0.02, 0.15)), waves=int(r.integers(1, 7)))


def _probe(m, c):
    """Weights of a pressure difference between two gauges under water."""
    C = m["C"]
    w = [m["V"] * torch.exp(-((C[0] - x * c["lx"]) ** 2 + (C[1] - 0.25 * c["ly"]) ** 2) / (0.1 * c["ly"]) ** 2)
         for x in (0.3, 0.7)]
    return (w[0] / w[0].sum() - w[1] / w[1].sum()).contiguous()


class _Mesh:
    def __init__(self, m):
        self.owner, self.neighbour, self.Sf, self.C = m["owner"], m["neighbour"], m["Sf"], m["C"]


def _cell_sum(n, o, v, at_o, at_v):
    """Face values summed to their owners and neighbours, in the same order
    every time (a cell has one face in each of its six directions)."""
    out = torch.zeros(n, device=DEV, dtype=F64)
    step = v - o
    for s in torch.unique(step).tolist():
        k = step == s
        out[o[k]] += at_o[k]
        out[v[k]] += at_v[k]
    return out


def _csr(o, v, gam, n, ref):
    """The pinned GFM system as CSR on the device."""
    diag = _cell_sum(n, o, v, gam, gam)
    diag[ref] *= 2.0
    i = torch.arange(n, device=DEV)
    rows, cols = torch.cat([i, o, v]), torch.cat([i, v, o])
    vals = torch.cat([diag, -gam, -gam])
    order = torch.argsort(rows * n + cols)
    ptr = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return ptr.to(torch.int32), cols[order].to(torch.int32), vals[order].contiguous()


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        qs = [_problem(_tank_case(c, t, seed), 1000 * seed + t) for t in range(c["tanks"])]
        h = gfm.GFMBatch([_Mesh(q["m"]) for q in qs], renumber=c["renumber"])
        return dict(case=c, h=h, alpha=torch.cat([q["alpha"] for q in qs]), phi=torch.cat([q["phi"] for q in qs]),
                    phys=[q["phys"] for q in qs])
    if kind == "nonorth":
        g = _gen(seed)
        m = _wavy(c["nx"], c["ny"], c["eps"])
        level = 0.4 + 0.2 * torch.rand(1, device=DEV, generator=g, dtype=F64)
        q = dict(m=m, g=g, alpha=((level - m["C"][1]) / m["h"][1] + 0.5).clamp(0.0, 1.0).contiguous())
        h = _handle(m, c)
        h.assemble(q["alpha"], _flux(m, g), RHO_W, RHO_A, GRAV, 0, 0.0)
        return dict(case=c, h=h, p=_pressure_like(m, q), V=m["V"].contiguous(), xf=m["xf"].contiguous())
    if kind == "iso":
        g = _gen(seed)
        m = _graded(c["nx"], c["ny"], c["nz"], g)
        n = m["n"]
        rnd = lambda *s: torch.rand(s, device=DEV, generator=g, dtype=F64)  # noqa: E731
        # an interface through about a tenth of the cells, as near a surface
        has = (rnd(n) < 0.1).to(torch.int8)
        nS = 2.0 * rnd(3, n) - 1.0
        nS = (nS / nS.norm(dim=0)).contiguous()
        xS = (m["C"] + 0.3 * (rnd(3, n) - 0.5) * m["V"].pow(1 / 3)).contiguous()
        UnS = (rnd(n) - 0.5).contiguous()
        phi = ((rnd(m["F"]) - 0.5) * m["Sf"].norm(dim=0)).contiguous()
        dt = 0.4 * min(m["h"])
        return dict(case=c, h=_handle(m, c), a=(rnd(n), phi, dt, m["fv_ptr"], m["fv_xyz"], m["xf"].contiguous(), has, xS,
                                                nS, UnS, m["V"].contiguous()))
    q = _problem(c, seed)
    m = q["m"]
    if kind == "csr":
        gam, J, _, _ = _face_quantities(m["owner"], m["neighbour"], m["Sf"], m["C"], q["alpha"])
        ptr, col, val = _csr(m["owner"], m["neighbour"], gam, m["n"], q["ref"])
        s = q["phi"] + gam * J
        b = _cell_sum(m["n"], m["owner"], m["neighbour"], -s, s)
        return dict(case=c, A=(ptr, col, val, b))
    st = dict(case=c, h=_handle(m, c), alpha=q["alpha"], phi=q["phi"], phys=q["phys"])
    if kind == "host":
        st["host"] = (q["alpha"].cpu().pin_memory(), q["phi"].cpu().pin_memory(),
                      torch.zeros(m["n"], dtype=F64).pin_memory())
    elif kind == "step":
        st["phis"] = _correctors(q, c["solves"])
        st["p"] = torch.zeros(m["n"], device=DEV, dtype=F64)
        st["info"] = torch.zeros(4 * c["solves"], device=DEV, dtype=F64)
    elif kind == "adjoint":
        st["w"] = _probe(m, c)
        st["alpha"].requires_grad_(True)
        st["phi"].requires_grad_(True)
    elif kind == "gradient":
        st["h"].assemble(q["alpha"], q["phi"], **q["phys"])
        st.update(p=_pressure_like(m, q), V=m["V"].contiguous(), xf=m["xf"].contiguous())
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "csr":
        x, _ = gfm.solve_csr_noalloc(*state["A"], rtol=c["rtol"])
        return x
    h = state["h"]
    if kind == "solve":
        h.assemble(state["alpha"], state["phi"], **state["phys"])
        return h.solve(mode=c["mode"], rtol=c["rtol"])[0]
    if kind == "host":
        a, f, p = state["host"]
        h.solve_host(a, f, p, mode=c["mode"], rtol=c["rtol"], **state["phys"])
        return p
    if kind == "batch":
        h.assemble(state["alpha"], state["phi"], state["phys"])
        return h.solve(rtol=c["rtol"])[0]
    if kind == "step":
        h.piso_step(state["alpha"], state["phis"], state["p"], state["info"], mode=c["mode"], rtol=c["rtol"],
                    **state["phys"])
        return state["p"]
    if kind == "adjoint":
        a, f = state["alpha"], state["phi"]
        p = gfm.GFMSolve.apply(a, f, h, state["phys"], dict(mode=c["mode"], rtol=c["rtol"]))
        ga, gf = torch.autograd.grad((state["w"] * p).sum(), (a, f))
        return p.detach(), ga, gf
    if kind == "assemble":
        h.assemble(state["alpha"], state["phi"], **state["phys"])
        return h.export_system()
    if kind == "gradient":
        return h.gradient(state["p"], state["V"], xf=state["xf"], phi=state["phi"])
    if kind == "nonorth":
        return h.nonorth_correct(state["p"], state["V"], xf=state["xf"], return_corr=True)
    return h.iso_advect(*state["a"][:-1], V=state["a"][-1])


def _faces_of(nx, ny, nz):
    return (nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1)


def work(case):
    """Each input read once and each output written once (plus, for a solve,
    nothing per iteration: how many iterations it takes is the solver's)."""
    c, kind = case, case["kind"]
    if kind == "batch":
        ts = [_tank_case(c, t, 0) for t in range(c["tanks"])]
        n = sum(t["nx"] * t["ny"] for t in ts)
        F = sum(_faces_of(t["nx"], t["ny"], 1) for t in ts)
    else:
        nz = c.get("nz", 1)
        n, F = c["nx"] * c["ny"] * nz, _faces_of(c["nx"], c["ny"], nz)
    mesh = F * (8 + 24) + n * 24  # owner, neighbour, S_f and the cell centres
    if kind == "csr":
        nnz = n + 2 * F
        return dict(bytes=12.0 * nnz + 4 * n + 16.0 * n, flops=2.0 * nnz)
    if kind in ("solve", "host", "batch"):
        return dict(bytes=mesh + 16.0 * n + 8.0 * F, flops=30.0 * F + 10.0 * n)
    if kind == "step":
        return dict(bytes=mesh + 16.0 * n + 8.0 * F * c["solves"], flops=(30.0 * F + 10.0 * n) * c["solves"])
    if kind == "adjoint":
        return dict(bytes=2.0 * mesh + 48.0 * n + 24.0 * F, flops=90.0 * F)
    if kind == "assemble":
        return dict(bytes=mesh + 24.0 * n + 32.0 * F, flops=30.0 * F)
    if kind == "gradient":
        return dict(bytes=mesh + 16.0 * n + 48.0 * n + 24.0 * F + 24.0 * F, flops=60.0 * F)
    if kind == "nonorth":
        return dict(bytes=mesh + 16.0 * n + 24.0 * F + 32.0 * F + 8.0 * F, flops=90.0 * F)
    return dict(bytes=F * (8.0 + 8 + 24 + 4 + 96 + 16) + n * (8.0 + 1 + 48 + 8 + 8 + 8), flops=20.0 * F + 8000.0 * 0.1 * F)


# ---------------------------------------------------------------------------
# what the paper's formulas give in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _face_quantities(o, v, S, C, alpha):
    """gamma, oriented jump, lambda and the wet side (+1 owner, -1 neighbour, 0 no interface) of each face."""
    ao, an = alpha[o], alpha[v]
    wo, wn = ao >= 0.5, an >= 0.5
    side = torch.where(wo == wn, 0, torch.where(wo, 1, -1))
    aW, aD = torch.where(wo, ao, an), torch.where(wo, an, ao)
    lam = torch.where(side == 0, wo.to(F64), (aW - 0.5) / torch.where(side == 0, torch.ones_like(aW), aW - aD))
    d = C[:, v] - C[:, o]
    gam = (S * S).sum(0) / (S * d).sum(0) / (lam * RHO_W + (1.0 - lam) * RHO_A)
    cw, cd = torch.where(wo, C[1, o], C[1, v]), torch.where(wo, C[1, v], C[1, o])
    J = side.to(F64) * ((RHO_W - RHO_A) * GRAV[1]) * (cw + lam * (cd - cw))
    return gam, J, lam, side


def _solve64(m, gam, rhs, ref, tol=2e-14, most=60_000):
    """Jacobi-CG of the pinned system on the structured grid, restarted from
    the true residual until it no longer falls."""
    nx, ny, nz = m["dims"]
    o, ax = m["owner"], _faces(nx, ny, nz)[2]
    gs = []
    for a, step in ((0, 1), (1, nx), (2, nx * ny)):
        full = torch.zeros(m["n"], device=DEV, dtype=F64)
        full[o[ax == a]] = gam[ax == a]
        gs.append((full.view(nz, ny, nx), 2 - a))
    use = [(f.narrow(dim, 0, f.shape[dim] - 1).contiguous(), dim) for f, dim in gs if f.shape[dim] > 1]
    diag = torch.zeros((nz, ny, nx), device=DEV, dtype=F64)
    for f, dim in use:
        k = f.shape[dim]
        diag.narrow(dim, 0, k).add_(f)
        diag.narrow(dim, 1, k).add_(f)
    pin = float(diag.view(-1)[ref])
    diag.view(-1)[ref] *= 2.0

    def mul(x):
        y = torch.zeros_like(x)
        for f, dim in use:
            k = f.shape[dim]
            t = f * (x.narrow(dim, 1, k) - x.narrow(dim, 0, k))
            y.narrow(dim, 0, k).sub_(t)
            y.narrow(dim, 1, k).add_(t)
        y.view(-1)[ref] += pin * x.view(-1)[ref]
        return y

    b = rhs.view(nz, ny, nx)
    x, bn, last, done, best = torch.zeros_like(b), float(b.norm()), math.inf, 0, None
    for _ in range(12):
        r = b - mul(x)
        rn = float(r.norm())
        if rn < last:
            best = x.clone()
        if rn <= tol * bn or rn > 0.5 * last or done >= most:
            break
        last = rn
        z = r / diag
        p, rz, it = z.clone(), (r * z).sum(), 0
        while done < most:
            s = mul(p)
            al = rz / (p * s).sum()
            x = x + al * p
            r = r - al * s
            z = r / diag
            rz1 = (r * z).sum()
            p = z + (rz1 / rz) * p
            rz = rz1
            done, it = done + 1, it + 1
            if it % 50 == 0 and float(r.norm()) <= max(0.3 * tol * bn, 1e-9 * rn):
                break
    return best.reshape(-1)


def _source(m, gam, J, phi):
    s = phi + gam * J
    return torch.zeros(m["n"], device=DEV, dtype=F64).index_add_(0, m["owner"], -s).index_add_(0, m["neighbour"], s)


def _to_caller(q, x):
    if "perm" not in q["m"]:
        return x
    out = torch.empty_like(x)
    out[q["m"]["perm"]] = x
    return out


def _gradient64(m, alpha, p, phi, V, xf):
    o, v, S, C = m["owner"], m["neighbour"], m["Sf"], m["C"]
    _, J, lam, _ = _face_quantities(o, v, S, C, alpha)
    rf = lam * RHO_W + (1.0 - lam) * RHO_A
    sd = (S * (C[:, v] - C[:, o])).sum(0)
    dp = (p[v] - p[o] - J) / rf
    w_o = (S * (xf - C[:, o])).sum(0) / sd
    G, U = torch.zeros((3, m["n"]), device=DEV, dtype=F64), torch.zeros((3, m["n"]), device=DEV, dtype=F64)
    for k in range(3):
        G[k].index_add_(0, o, w_o * dp * S[k]).index_add_(0, v, (1.0 - w_o) * dp * S[k])
        if phi is not None:
            U[k].index_add_(0, o, phi * (xf[k] - C[k, o])).index_add_(0, v, -phi * (xf[k] - C[k, v]))
    return G / V, U / V


def _iso64(case, seed):
    """The swept fraction of every face, triangle by triangle, integrated in time."""
    st = prepare(case, seed)
    m = _graded(case["nx"], case["ny"], case["nz"], _gen(seed))
    alpha, phi, dt, _, xyz, xf, has, xS, nS, UnS, V = st["a"]
    o, v = m["owner"], m["neighbour"]
    U = torch.where(phi >= 0, o, v)
    xs, ns, un = xS[:, U], nS[:, U], UnS[U]
    vert = xyz.reshape(3, -1, 4)
    cross = lambda a, b: torch.linalg.cross(a, b, dim=0).norm(dim=0)  # noqa: E731
    area, acc = torch.zeros_like(phi), torch.zeros_like(phi)
    for e in range(4):
        tri = torch.stack([xf, vert[:, :, e], vert[:, :, (e + 1) % 4]])  # [3 points][3][F]
        t, order = torch.sort(((tri - xs) * ns).sum(1) / un, dim=0)
        tri = torch.gather(tri, 0, order[:, None].expand(-1, 3, -1))
        x21, x31 = tri[1] - tri[0], tri[2] - tri[0]
        A = cross(tri[2] - tri[0], tri[1] - tri[0])
        t1, t2, t3 = t
        a2 = cross((t2 - t1) / (t3 - t1) * x31, x21) / A
        clip = lambda s, a, b: torch.minimum(torch.maximum(torch.full_like(a, s), a), b)  # noqa: E731
        lo, hi = clip(0.0, t1, t2), clip(dt, t1, t2)
        I = a2 * ((hi - t1) ** 3 - (lo - t1) ** 3) / (3.0 * (t2 - t1) ** 2)
        lo, hi = clip(0.0, t2, t3), clip(dt, t2, t3)
        I = I + (hi - lo) - (1.0 - a2) * ((t3 - lo) ** 3 - (t3 - hi) ** 3) / (3.0 * (t3 - t2) ** 2)
        I = I + (dt - t3.clamp_min(0.0)).clamp_min(0.0)
        area += A
        acc += A * torch.where(un < 0, dt - I, I)
    I = torch.where(has[U] != 0, acc / area, alpha[U] * dt)
    dV = phi * I
    out = torch.zeros_like(alpha).index_add_(0, o, dV).index_add_(0, v, -dV)
    return dV, I, alpha - out / V


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "iso":
        return _iso64(c, seed)
    if kind == "batch":
        if c["tanks"] > 16:
            return None
        out = []
        for t in range(c["tanks"]):
            q = _problem(_tank_case(c, t, seed), 1000 * seed + t)
            gam, J, _, _ = _face_quantities(q["u"]["owner"], q["u"]["neighbour"], q["u"]["Sf"], q["u"]["C"], q["a_u"])
            out.append(_solve64(q["u"], gam, _source(q["u"], gam, J, q["f_u"]), q["ref"], most=12_000))
        return torch.cat(out)
    if kind == "nonorth":
        s = prepare(c, seed)
        g = _gen(seed)
        m = _wavy(c["nx"], c["ny"], c["eps"])
        level = 0.4 + 0.2 * torch.rand(1, device=DEV, generator=g, dtype=F64)
        alpha = ((level - m["C"][1]) / m["h"][1] + 0.5).clamp(0.0, 1.0)
        G, _ = _gradient64(m, alpha, s["p"], None, m["V"], m["xf"])
        o, v, S, C = m["owner"], m["neighbour"], m["Sf"], m["C"]
        d = C[:, v] - C[:, o]
        sd = (S * d).sum(0)
        w_o = (S * (C[:, v] - m["xf"])).sum(0) / sd
        k = S - ((S * S).sum(0) / sd) * d
        return (k * (w_o * G[:, o] + (1.0 - w_o) * G[:, v])).sum(0)
    q = _problem(c, seed)
    u, m = q["u"], q["m"]
    if kind == "assemble":
        gam, J, lam, _ = _face_quantities(m["owner"], m["neighbour"], m["Sf"], m["C"], q["alpha"])
        diag = torch.zeros(m["n"], device=DEV, dtype=F64).index_add_(0, m["owner"], gam).index_add_(0, m["neighbour"], gam)
        diag[q["phys"]["ref_cell"]] *= 2.0
        return {"lambda": lam, "gamma": gam, "jump": J, "diag": diag, "b": _source(m, gam, J, q["phi"])}
    if kind == "gradient":
        return _gradient64(m, q["alpha"], _pressure_like(m, q), q["phi"], m["V"], m["xf"])
    gam, J, lam, side = _face_quantities(u["owner"], u["neighbour"], u["Sf"], u["C"], q["a_u"])
    phi = q["f_u"]
    if kind == "step":
        phi = _correctors(dict(q, m=u, phi=q["f_u"]), c["solves"])[-1]
    p = _solve64(u, gam, _source(u, gam, J, phi), q["ref"])
    if kind == "host":
        return _to_caller(q, p).cpu()
    if kind != "adjoint":
        return _to_caller(q, p)
    C, o, v = u["C"], u["owner"], u["neighbour"]
    mu = _solve64(u, gam, _probe(u, c), q["ref"])
    dmu = mu[o] - mu[v]
    face = side != 0
    a = q["a_u"]
    W, D = torch.where(side >= 0, o, v), torch.where(side >= 0, v, o)
    rf = lam * RHO_W + (1.0 - lam) * RHO_A
    dgam = -gam * (RHO_W - RHO_A) / rf
    dJ = side.to(F64) * ((RHO_W - RHO_A) * GRAV[1]) * (C[1, D] - C[1, W])
    dlam = torch.where(face, -dmu * (p[o] - p[v] + J) * dgam - gam * dmu * dJ, torch.zeros_like(dmu))
    den = torch.where(face, (a[W] - a[D]) ** 2, torch.ones_like(dmu))
    ga = torch.zeros_like(a).index_add_(0, W, dlam * (0.5 - a[D]) / den).index_add_(0, D, dlam * (a[W] - 0.5) / den)
    return p, ga, -dmu
