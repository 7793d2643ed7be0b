"""Performance cases: the work a user of this library has it do, through its public Python API.

A case is a plain dict.  `kind` is the pass that is measured:
  spmv      y = A x with the assembled matrix (a caller's own Krylov loop)
  assemble  mesh, plies or permeability -> the BSR system on the device
  precond   z = M^-1 r, FP64 two-level Schwarz with the zero-energy-mode coarse space
  resident  a new load on a resident preconditioner, then the Krylov solve
  batch     one batched solve of several uneven set-up blocks
  whole     assembly, preconditioner set-up and solve: time to solution
`physics` is the layered-composite elasticity block or the scalar Darcy problem, `prec` the
precision of the subdomain factors.  Solves run to the default relative residual, 1e-8.
"""
import math

import numpy as np
import torch

import paper_1901_05188_gb300 as pkg

# ply and resin constants of the layered composite (MPa), layer thicknesses and in-plane
# element edge (mm)
PLY = (162000.0, 10000.0, 10000.0, 5200.0, 5200.0, 3500.0, 0.35, 0.35, 0.5)
RESIN = (10000.0,) * 3 + (10000.0 / 2.7,) * 3 + (0.35,) * 3
PLY_T, RESIN_T, EDGE = 0.23, 0.02, 0.5
CELL = (20.0, 10.0, 2.0)          # Darcy cell edges (ft)
TOL = 1e-8
PREC = {"fp64": pkg.GENEO_FP64, "mixed": pkg.GENEO_MIXED_FP32}


# ---- the cases -----------------------------------------------------------------------

def _case(kind, physics, n, parts, prec="fp64", plies=4, resin=False, wrinkle=False, **more):
    return dict(kind=kind, physics=physics, nx=n[0], ny=n[1], nz=n[2], px=parts[0], py=parts[1],
                pz=parts[2], prec=prec, plies=plies, resin=resin, wrinkle=wrinkle, **more)


def listed():
    return [
        # the smallest call: one product with an 8x8x8 block's matrix
        dict(_case("spmv", "elastic", (8, 8, 8), (1, 1, 1)), name="spmv_8x8x8"),
        # the same product on the 1.2 M unknown wrinkled laminate
        dict(_case("spmv", "elastic", (128, 64, 48), (1, 1, 1), plies=24, wrinkle=True),
             name="spmv_128x64x48"),
        # a new design (stacking sequence) of the large laminate, assembled
        dict(_case("assemble", "elastic", (128, 64, 48), (1, 1, 1), plies=24, wrinkle=True),
             name="assemble_128x64x48"),
        # a new permeability realisation on the SPE10 grid, assembled
        dict(_case("assemble", "darcy", (60, 220, 85), (1, 1, 1)), name="assemble_darcy_60x220x85"),
        # one preconditioner application (a caller's own Krylov loop), FP64 factors
        dict(_case("precond", "elastic", (64, 32, 24), (4, 4, 2), plies=12, resin=True),
             name="precond_fp64_64x32x24"),
        # a small coupon answered from its resident factors: launch and latency bound
        dict(_case("resident", "elastic", (8, 8, 8), (2, 2, 2), plies=4, modes=6),
             name="resident_fp64_8x8x8"),
        # a new load case on a resident FP64 preconditioner, ragged parts
        dict(_case("resident", "elastic", (57, 35, 23), (4, 4, 2), plies=9, resin=True),
             name="resident_fp64_57x35x23"),
        # the large laminate answered from its resident mixed-precision factors
        dict(_case("resident", "elastic", (128, 64, 48), (8, 4, 4), "mixed", plies=24, wrinkle=True),
             name="resident_mixed_128x64x48"),
        # eight uneven blocks solved together
        dict(kind="batch", physics="elastic", blocks=8, el_lo=8000, el_hi=24000, sizes=3,
             prec="mixed", name="batch_mixed_8"),
        # time to solution, all FP64, the 12-ply laminate with resin interlayers
        dict(_case("whole", "elastic", (64, 32, 24), (4, 4, 2), plies=12, resin=True),
             name="whole_fp64_64x32x24"),
        # time to solution of a large wrinkled laminate, mixed precision
        dict(_case("whole", "elastic", (96, 48, 48), (6, 3, 4), "mixed", plies=24, wrinkle=True),
             name="whole_mixed_96x48x48"),
        # time to solution of one permeability realisation on the SPE10 grid, mixed precision
        dict(_case("whole", "darcy", (60, 220, 85), (6, 18, 1), "mixed"),
             name="whole_darcy_mixed_60x220x85"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _block(rng, most, parts):
    """A laminated block of up to `most` elements; `parts`: split into boxes of about 16x10x12."""
    resin = rng.random() < 0.5
    plies = rng.randint(3, 12)
    nz = 2 * plies - 1 if resin else plies * rng.randint(1, 3)
    area = max(36, _log_int(rng, 300, most) // nz)
    nx = max(6, int(round(math.sqrt(area * rng.uniform(1.0, 3.0)))))
    ny = max(6, area // nx)
    p = tuple(max(1, round(n / s)) for n, s in zip((nx, ny, nz), (16, 10, 12)))
    if p == (1, 1, 1):
        p = (2, 1, 1)
    return (nx, ny, nz), (p if parts else (1, 1, 1)), dict(plies=plies, resin=resin,
                                                          wrinkle=rng.random() < 0.5)


def _darcy(rng, most, parts):
    """A Darcy grid in about SPE10's proportions, split in-plane over the full height."""
    n = _log_int(rng, 1000, most)
    nx = max(6, int(round((n * rng.uniform(0.15, 0.4)) ** (1 / 3) * 0.9)))
    nz = max(6, int(round(nx * rng.uniform(0.8, 1.6))))
    ny = max(6, n // (nx * nz))
    p = (max(1, round(nx / 10)), max(1, round(ny / 12)), 1)
    if p == (1, 1, 1):
        p = (1, 2, 1)
    return (nx, ny, nz), (p if parts else (1, 1, 1)), {}


def draw(rng):
    kind = rng.choice(["spmv", "assemble", "precond", "resident", "resident", "batch", "whole", "whole"])
    if kind == "batch":
        return dict(kind=kind, physics="elastic", blocks=rng.randint(2, 8), el_lo=2000,
                    el_hi=rng.randint(6000, 20000), sizes=rng.randint(0, 10 ** 6),
                    prec=rng.choice(["mixed", "fp64"]))
    physics = "elastic" if kind == "precond" else rng.choice(["elastic", "elastic", "darcy"])
    prec = rng.choice(["mixed", "fp64"]) if kind in ("resident", "whole") else "fp64"
    if kind in ("spmv", "assemble"):
        n, parts, more = (_darcy(rng, 1_000_000, False) if physics == "darcy"
                          else _block(rng, 380_000, False))
    elif physics == "darcy":
        n, parts, more = _darcy(rng, 300_000, True)
    else:
        n, parts, more = _block(rng, 40_000 if kind == "precond" else 90_000, True)
    return _case(kind, physics, n, parts, prec, **more)


# ---- inputs --------------------------------------------------------------------------

def _layers(nz, plies, resin, angles):
    """Node heights, material and ply angle (degrees) of nz element layers: plies of equal
    thickness with one-element resin interlayers, the lowest plies one element taller where
    the split is uneven."""
    n_res = plies - 1 if resin else 0
    base, extra = divmod(nz - n_res, plies)
    dz, mat, ang = [], [], []
    for p in range(plies):
        k = base + (p < extra)
        dz += [PLY_T / k] * k
        mat += [0] * k
        ang += [float(angles[p])] * k
        if resin and p + 1 < plies:
            dz.append(RESIN_T)
            mat.append(1)
            ang.append(0.0)
    return np.concatenate([[0.0], np.cumsum(dz)]), np.array(mat), np.array(ang)


def _laminate(c, seed):
    rs = np.random.RandomState(seed % (1 << 31))
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    z, mat, ang = _layers(nz, c["plies"], c["resin"], rs.choice([0.0, 45.0, -45.0, 90.0], c["plies"]))
    x, y = np.arange(nx + 1) * EDGE, np.arange(ny + 1) * EDGE
    dev = dict(device="cuda")
    layer = torch.arange(nz, **dev).repeat_interleave(nx * ny)
    mat_t = torch.tensor(mat, dtype=torch.int32, **dev)[layer].contiguous()
    theta = torch.deg2rad(torch.tensor(ang, dtype=torch.float64, **dev))[layer].contiguous()
    phi = torch.zeros_like(theta)
    if c["wrinkle"]:                 # out-of-plane fibre wrinkle about a seeded centre
        xc = (torch.arange(nx, dtype=torch.float64, **dev) + 0.5 - nx * rs.uniform(0.4, 0.6)) / 10.0
        yc = (torch.arange(ny, dtype=torch.float64, **dev) + 0.5 - ny * rs.uniform(0.4, 0.6)) / 10.0
        bump = math.radians(8.0) * torch.exp(-0.5 * (xc[None, :] ** 2 + yc[:, None] ** 2))
        phi = torch.where(mat_t == 1, phi, bump.reshape(-1).repeat(nz)).contiguous()
    clamped = torch.arange(0, (nx + 1) * (ny + 1) * (nz + 1), nx + 1, **dev)
    dofs = (3 * clamped[:, None] + torch.arange(3, **dev)).reshape(-1).to(torch.int32)
    modes = (dict(fixed_modes=c["modes"], threshold=0.0, max_modes=20, shift=-0.01) if c.get("modes")
             else dict(fixed_modes=0, threshold=0.0, max_modes=20, shift=-0.01))
    return dict(nx=nx, ny=ny, nz=nz, x=x, y=y, z=z, materials=np.array([PLY, RESIN]),
                elem_mat=mat_t, elem_theta=theta, elem_phi=phi, dirichlet_dofs=dofs,
                dirichlet_values=torch.zeros(dofs.numel(), dtype=torch.float64, **dev),
                top_pressure=float(rs.uniform(0.5, 2.0)), nodal_load=None,
                partition=(c["px"], c["py"], c["pz"], 1), modes=modes)


def _permeability(nx, ny, nz, seed):
    """Log-normal permeability correlated over about 20 cells in-plane and 2 vertically, every
    third layer a meandering channel in a tight background; Kz = 0.1 Kx."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.fft.fftn(torch.randn(nz, ny, nx, dtype=torch.float64, device="cuda", generator=g))
    for axis, (n, ell) in enumerate(((nz, 2.0), (ny, 20.0), (nx, 20.0))):
        k = torch.fft.fftfreq(n, dtype=torch.float64, device="cuda")
        shape = [1, 1, 1]
        shape[axis] = n
        f = f * torch.exp(-0.5 * (2 * math.pi * k * ell) ** 2).reshape(shape)
    field = torch.fft.ifftn(f).real
    logk = -1.0 + 1.5 * (field - field.mean()) / field.std()
    layers = torch.arange(1, nz, 3, device="cuda")
    rows = torch.arange(ny, dtype=torch.float64, device="cuda")
    centre = nx / 2 + 0.3 * nx * torch.sin(2 * math.pi * rows / ny + layers[:, None].double())
    inside = (torch.arange(nx, device="cuda").double() - centre[:, :, None]).abs() < 2.0
    logk[1::3] = torch.where(inside, 2.0, -4.0).double()
    kx = (10.0 ** logk).reshape(-1)
    return torch.stack([kx, kx, 0.1 * kx], dim=1).contiguous()


def _reservoir(c, seed):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    bottom = torch.arange((nx + 1) * (ny + 1), dtype=torch.int32, device="cuda")
    return dict(kind="darcy", nx=nx, ny=ny, nz=nz, x=np.arange(nx + 1) * CELL[0],
                y=np.arange(ny + 1) * CELL[1], z=np.arange(nz + 1) * CELL[2],
                perm=_permeability(nx, ny, nz, seed), dirichlet_dofs=bottom,
                dirichlet_values=torch.zeros(bottom.numel(), dtype=torch.float64, device="cuda"),
                source=1.0, nodal_load=None, partition=(c["px"], c["py"], c["pz"], 1),
                modes=dict(fixed_modes=0, threshold=0.0, max_modes=20, shift=-0.01))


def _problem(c, seed):
    return _reservoir(c, seed) if c["physics"] == "darcy" else _laminate(c, seed)


def _load(c, p, seed):
    """A smooth seeded nodal load (elasticity) or a scattered source (Darcy)."""
    g = torch.Generator(device="cuda").manual_seed(seed + 77)
    n = (p["nx"] + 1) * (p["ny"] + 1) * (p["nz"] + 1)
    nc = 1 if c["physics"] == "darcy" else 3
    return 1e-2 * torch.randn(nc * n, dtype=torch.float64, device="cuda", generator=g)


def _batch_cases(c):
    rs = np.random.RandomState(c["sizes"])
    out = []
    for _ in range(c["blocks"]):
        n_el = math.exp(rs.uniform(math.log(c["el_lo"]), math.log(c["el_hi"])))
        plies = int(rs.randint(4, 13))
        nz = plies * int(rs.randint(1, 3))
        nx = max(8, int(round(math.sqrt(n_el / nz * rs.uniform(1.0, 3.0)))))
        ny = max(8, int(round(n_el / nz / nx)))
        parts = (max(2, round(nx / 14)), max(1, round(ny / 12)), max(1, round(nz / 14)))
        out.append(_case("batch", "elastic", (nx, ny, nz), parts, c["prec"], plies=plies))
    return out


def _set_up(c, p):
    s = pkg.GeneoSolver()
    s.assemble(p)
    coarse = pkg.GENEO_COARSE_ZEM if c["kind"] == "precond" else pkg.GENEO_COARSE_GENEO
    s.setup(p, PREC[c["prec"]], pkg.GENEO_AS, coarse)
    return s


def prepare(case, seed):
    if case["kind"] == "batch":
        solvers = []
        for i, c in enumerate(_batch_cases(case)):
            solvers.append(_set_up(c, _laminate(c, seed + 1000 * i)))
        outs = [torch.empty(s.ndof, dtype=torch.float64, device="cuda") for s in solvers]
        return dict(case=case, solvers=solvers, batch=pkg.GeneoBatch(solvers), outs=outs)
    p = _problem(case, seed)
    st = dict(case=case, p=p)
    if case["kind"] in ("assemble", "whole"):
        st["solver"] = pkg.GeneoSolver()
        if case["kind"] == "whole":
            nc = 1 if case["physics"] == "darcy" else 3
            n = nc * (p["nx"] + 1) * (p["ny"] + 1) * (p["nz"] + 1)
            st["out"] = torch.empty(n, dtype=torch.float64, device="cuda")
        else:
            nc2 = 1 if case["physics"] == "darcy" else 9
            nn = (p["nx"] + 1) * (p["ny"] + 1) * (p["nz"] + 1)
            nb = (3 * p["nx"] + 1) * (3 * p["ny"] + 1) * (3 * p["nz"] + 1)
            st["system"] = (torch.empty(nn + 1, dtype=torch.int32, device="cuda"),
                            torch.empty(nb, dtype=torch.int32, device="cuda"),
                            torch.empty(nc2 * nb, dtype=torch.float64, device="cuda"),
                            torch.empty(nn * (1 if nc2 == 1 else 3), dtype=torch.float64, device="cuda"))
        return st
    if case["kind"] == "spmv":
        st["solver"] = pkg.GeneoSolver()
        st["solver"].assemble(p)
    else:
        st["solver"] = _set_up(case, p)
    if case["kind"] == "resident":
        st["load"] = _load(case, p, seed)
        st["out"] = torch.empty(st["solver"].ndof, dtype=torch.float64, device="cuda")
    else:
        g = torch.Generator(device="cuda").manual_seed(seed + 5)
        st["x"] = torch.randn(st["solver"].ndof, dtype=torch.float64, device="cuda", generator=g)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        st["batch"].solve(TOL, outs=st["outs"])
        return st["outs"]
    s = st["solver"]
    if kind == "spmv":
        return s.spmv(st["x"])
    if kind == "precond":
        return s.apply_preconditioner(st["x"])
    if kind == "assemble":
        s.assemble(st["p"])
        pkg.geneo_get_system(s.ctx, *st["system"])
        return st["system"]
    if kind == "resident":
        s.set_load(st["load"], 1.0)
    else:
        s.assemble(st["p"])
        s.setup(st["p"], PREC[case["prec"]])
    s.solve(TOL, out=st["out"])
    return st["out"]


# ---- work ----------------------------------------------------------------------------

def _axis(n, p):
    """Element boxes of overlap 1 and interior node ranges (inclusive) of one axis."""
    out = []
    for k in range(p):
        lo, hi = max(0, k * n // p - 1), min(n, (k + 1) * n // p + 1)
        out.append((lo, hi, lo + (lo > 0), hi - (hi < n)))
    return out


def _bands(c, nc):
    """(unknowns, half-bandwidth) of every subdomain's interior and Neumann matrix, longest
    axis numbered slowest."""
    def band(n):
        a, b, _ = sorted(n)
        return nc * n[0] * n[1] * n[2], nc * (1 + a + a * b) + nc - 1
    boxes = [_axis(c[k], c[q]) for k, q in (("nx", "px"), ("ny", "py"), ("nz", "pz"))]
    inner, neu = [], []
    for x in boxes[0]:
        for y in boxes[1]:
            for z in boxes[2]:
                inner.append(band([b[3] - b[2] + 1 for b in (x, y, z)]))
                neu.append(band([b[1] - b[0] + 1 for b in (x, y, z)]))
    return inner, neu


def work(case):
    """Least work of one pass.  Solves: one pass over the matrix and the factors (their number of
    iterations is the method's affair); set-ups: the factorisations too."""
    if case["kind"] == "batch":
        ws = [work(dict(c, kind="resident")) for c in _batch_cases(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    nc = 1 if case["physics"] == "darcy" else 3
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nc * (nx + 1) * (ny + 1) * (nz + 1)
    nb = (3 * nx + 1) * (3 * ny + 1) * (3 * nz + 1)
    matrix = nb * (8 * nc * nc + 4) + 4 * n // nc
    kind = case["kind"]
    if kind == "spmv":
        return dict(bytes=matrix + 16 * n, flops=2 * nc * nc * nb)
    if kind == "assemble":
        el = nx * ny * nz
        return dict(bytes=matrix + 8 * n + el * (24 if nc == 1 else 20), flops=64 * (10 if nc == 1 else 170) * el)
    inner, neu = _bands(case, nc)
    esz = 4 if case["prec"] == "mixed" else 8
    entries = sum(m * (b + 1) - b * (b + 1) // 2 for m, b in inner)
    out = dict(bytes=2 * entries * esz + 16 * n, flops=4 * entries)
    if kind in ("resident", "whole"):
        out["bytes"] += matrix
        out["flops"] += 2 * nc * nc * nb
    if kind == "whole":
        for m, b in inner + neu:
            out["flops"] += max(m - b, 0) * b * b + b * b * b // 3
        out["bytes"] += sum(m * (b + 1) for m, b in neu) * 8
    return out


# ---- the same in 64 bits, plain torch ----------------------------------------------------

def _stiffness_laminate(p):
    """Element matrices (nel, 8, 3, 8, 3): orthotropic stiffness in ply axes as a fourth-order
    tensor, rotated by Rz(theta) Ry(phi), 2x2x2 Gauss points."""
    dev = dict(dtype=torch.float64, device="cuda")
    pairs = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
    base = []
    for E1, E2, E3, G12, G13, G23, n12, n13, n23 in p["materials"]:
        S = torch.zeros(6, 6, **dev)
        S[:3, :3] = torch.tensor([[1 / E1, -n12 / E1, -n13 / E1], [-n12 / E1, 1 / E2, -n23 / E2],
                                  [-n13 / E1, -n23 / E2, 1 / E3]], **dev)
        S[3, 3], S[4, 4], S[5, 5] = 1 / G23, 1 / G13, 1 / G12
        V = torch.linalg.inv(S)
        C = torch.zeros(3, 3, 3, 3, **dev)
        for a, (i, j) in enumerate(pairs):
            for b, (k, l) in enumerate(pairs):
                for u, v in {(i, j), (j, i)}:
                    for s, t in {(k, l), (l, k)}:
                        C[u, v, s, t] = V[a, b]
        base.append(C)
    t, f = p["elem_theta"], p["elem_phi"]
    o = torch.zeros_like(t)
    rz = torch.stack([t.cos(), -t.sin(), o, t.sin(), t.cos(), o, o, o, o + 1], 1).reshape(-1, 3, 3)
    ry = torch.stack([f.cos(), o, f.sin(), o, o + 1, o, -f.sin(), o, f.cos()], 1).reshape(-1, 3, 3)
    Q = rz @ ry
    C = torch.stack(base)[p["elem_mat"].long()]
    for _ in range(4):               # each rotation moves the next index to the back
        C = torch.einsum("eijkl,epi->ejklp", C, Q)
    h = _edges(p)
    K = torch.zeros(t.numel(), 8, 3, 8, 3, **dev)
    for grads, w in _gauss(h):
        K += torch.einsum("eaj,eijkl,ebl,e->eaibk", grads, C, grads, w)
    return K


def _stiffness_darcy(p):
    h = _edges(p)
    K = torch.zeros(h.shape[0], 8, 1, 8, 1, dtype=torch.float64, device="cuda")
    for grads, w in _gauss(h):
        K[:, :, 0, :, 0] += torch.einsum("eaj,ej,ebj,e->eab", grads, p["perm"], grads, w)
    return K


def _edges(p):
    d = [torch.tensor(np.diff(p[k]), device="cuda") for k in "xyz"]
    z, y, x = torch.meshgrid(d[2], d[1], d[0], indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)


def _gauss(h):
    corner = torch.tensor([[a & 1, a >> 1 & 1, a >> 2] for a in range(8)], dtype=torch.float64,
                          device="cuda")
    w = h.prod(1) / 8
    for q in range(8):
        pt = 0.5 + (corner[q] - 0.5) / math.sqrt(3.0)
        f = torch.where(corner == 1, pt, 1 - pt)              # (8, 3) factors per axis
        s = 2 * corner - 1
        g = torch.stack([s[:, 0] * f[:, 1] * f[:, 2], f[:, 0] * s[:, 1] * f[:, 2],
                         f[:, 0] * f[:, 1] * s[:, 2]], 1)
        yield g[None] / h[:, None, :], w


def _system(p):
    """Rows of A in 27 neighbour slots (nnode, 27, nc, nc), the slots' columns (-1 outside),
    the load and the Dirichlet mask."""
    darcy = p.get("kind") == "darcy"
    nc = 1 if darcy else 3
    nx, ny, nz = p["nx"], p["ny"], p["nz"]
    sx, sy = nx + 1, (nx + 1) * (ny + 1)
    nn = sy * (nz + 1)
    K = _stiffness_darcy(p) if darcy else _stiffness_laminate(p)
    dev = dict(device="cuda")
    ez, ey, ex = torch.meshgrid(*[torch.arange(n, **dev) for n in (nz, ny, nx)], indexing="ij")
    first = (ex + sx * ey + sy * ez).reshape(-1)
    val = torch.zeros(nn, 27, nc, nc, dtype=torch.float64, **dev)
    at = [(a & 1, a >> 1 & 1, a >> 2) for a in range(8)]
    for a in range(8):
        na = first + at[a][0] + sx * at[a][1] + sy * at[a][2]
        for b in range(8):
            d = [v - u + 1 for u, v in zip(at[a], at[b])]
            val[na, d[0] + 3 * d[1] + 9 * d[2]] += K[:, a, :, b, :]
    del K
    node = torch.arange(nn, **dev)
    i, j, k = node % sx, node // sx % (ny + 1), node // sy
    col = torch.full((nn, 27), -1, dtype=torch.int64, **dev)
    for s in range(27):
        u, v, w = i + s % 3 - 1, j + s // 3 % 3 - 1, k + s // 9 - 1
        ok = (u >= 0) & (u <= nx) & (v >= 0) & (v <= ny) & (w >= 0) & (w <= nz)
        col[:, s] = torch.where(ok, u + sx * v + sy * w, -1)
    mask = torch.zeros(nc * nn, dtype=torch.bool, **dev)
    mask[p["dirichlet_dofs"].long()] = True
    mask = mask.reshape(nn, nc)
    h = _edges(p)
    b = torch.zeros(nn, nc, dtype=torch.float64, **dev)
    if darcy:
        for a in range(8):
            b[first + at[a][0] + sx * at[a][1] + sy * at[a][2], 0] += p["source"] * h.prod(1) / 8
    else:
        area = h[:, 0] * h[:, 1] / 4
        top = ez.reshape(-1) == nz - 1
        for a in range(4, 8):
            na = first + at[a][0] + sx * at[a][1] + sy * at[a][2]
            b[na[top], 2] -= p["top_pressure"] * area[top]
    far = mask[col.clamp(min=0)]                              # (nn, 27, nc)
    drop = mask[:, None, :, None] | far[:, :, None, :]
    val = torch.where(drop, torch.zeros_like(val), val)
    val[:, 13] += torch.diag_embed(mask.double())
    return val, col, torch.where(mask, torch.zeros_like(b), b).reshape(-1), mask.reshape(-1)


def _csr(val, col):
    nn, _, nc, _ = val.shape
    keep = (col >= 0)[:, None, :, None].expand(nn, nc, 27, nc)
    c = (nc * col[:, None, :, None] + torch.arange(nc, device="cuda")).expand(nn, nc, 27, nc)[keep]
    count = (nc * (col >= 0).sum(1)).repeat_interleave(nc)
    ptr = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), count.cumsum(0)])
    return torch.sparse_csr_tensor(ptr, c, val.permute(0, 2, 1, 3)[keep], size=(nc * nn, nc * nn))


def _dense(val, col, nodes):
    """The rows and columns of `nodes` as a dense matrix."""
    nn, _, nc, _ = val.shape
    local = torch.full((nn + 1,), -1, dtype=torch.int64, device="cuda")
    local[nodes] = torch.arange(nodes.numel(), device="cuda")
    c = local[torch.where(col[nodes] < 0, nn, col[nodes])]    # (m, 27)
    row, slot = torch.nonzero(c >= 0, as_tuple=True)
    m = nodes.numel()
    A = torch.zeros(m, nc, m, nc, dtype=torch.float64, device="cuda")
    A[row, :, c[row, slot], :] = val[nodes][row, slot]
    return A.reshape(nc * m, nc * m)


def _solve(val, col, b):
    """A u = b: dense Cholesky with refinement, or diagonally scaled CG run to stagnation."""
    n = b.numel()
    A = _csr(val, col)
    if n <= 12000:
        L = torch.linalg.cholesky(_dense(val, col, torch.arange(val.shape[0], device="cuda")))
        u = torch.zeros_like(b)
        for _ in range(3):
            u += torch.cholesky_solve((b - A @ u)[:, None], L)[:, 0]
        return u
    d = val[:, 13].diagonal(dim1=1, dim2=2).reshape(-1)
    u = torch.zeros_like(b)
    for _ in range(2):               # restarted once on the true residual
        r = b - A @ u
        z = r / d
        q = z.clone()
        rz = r @ z
        for it in range(20000):
            Aq = A @ q
            alpha = rz / (q @ Aq)
            u = u + alpha * q
            r = r - alpha * Aq
            if it % 100 == 99 and float(r.norm()) <= 1e-14 * float(b.norm()):
                break
            z = r / d
            new = r @ z
            q = z + (new / rz) * q
            rz = new
    return u


def _precond(case, p, r):
    """z = sum_j R_j^T A_j^-1 R_j r + Z A_H^-1 Z^T r with the rigid displacements of every
    floating subdomain, unit length, weighted by the partition of unity, as Z."""
    val, col, _, mask = _system(p)
    sx, sy = p["nx"] + 1, (p["nx"] + 1) * (p["ny"] + 1)
    xyz = [torch.tensor(p[k], device="cuda") for k in "xyz"]
    boxes = [_axis(p[k], n) for k, n in zip(("nx", "ny", "nz"), p["partition"][:3])]
    subs = [(x, y, z) for z in boxes[2] for y in boxes[1] for x in boxes[0]]

    def nodes(lo, hi):
        k, j, i = torch.meshgrid(*[torch.arange(l, h + 1, device="cuda") for l, h in
                                   zip(lo[::-1], hi[::-1])], indexing="ij")
        return i.reshape(-1), j.reshape(-1), k.reshape(-1)

    def dofs(i, j, k):
        return (3 * (i + sx * j + sy * k)[:, None] + torch.arange(3, device="cuda")).reshape(-1)

    z = torch.zeros_like(r)
    count = torch.zeros_like(r)
    inner = []
    for s in subs:
        ijk = nodes([b[2] for b in s], [b[3] for b in s])
        g = dofs(*ijk)
        inner.append(g)
        count[g] += 1
        L = torch.linalg.cholesky(_dense(val, col, ijk[0] + sx * ijk[1] + sy * ijk[2]))
        z[g] += torch.cholesky_solve(r[g][:, None], L)[:, 0]
    cols = []
    for s, g in zip(subs, inner):
        i, j, k = nodes([b[0] for b in s], [b[1] for b in s])
        all_g = dofs(i, j, k)
        if bool(mask[all_g].any()):
            continue
        dx, dy, dz = (ax[t] - 0.5 * (ax[b[0]] + ax[b[1]]) for ax, t, b in zip(xyz, (i, j, k), s))
        o, e = torch.zeros_like(dx), torch.ones_like(dx)
        for v in ((e, o, o), (o, e, o), (o, o, e), (o, -dz, dy), (dz, o, -dx), (-dy, dx, o)):
            m = torch.zeros_like(r)
            m[all_g] = torch.stack(v, 1).reshape(-1)
            m = m / m.norm()
            out = torch.zeros_like(r)
            out[g] = m[g] / count[g]
            cols.append(torch.where(mask, torch.zeros_like(out), out))
    if cols:
        Z = torch.stack(cols, 1)
        AH = Z.T @ (_csr(val, col) @ Z)
        z = z + Z @ torch.linalg.solve(AH, Z.T @ r)
    return z


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i, c in enumerate(_batch_cases(case)):
            val, col, b, _ = _system(_laminate(c, seed + 1000 * i))
            out.append(_solve(val, col, b) if b.numel() <= 12000 else None)
        return out if any(v is not None for v in out) else None
    nc = 1 if case["physics"] == "darcy" else 3
    n = nc * (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    # a plain solver takes minutes on the largest systems, and loses the digits to compare on a
    # permeability contrast of 1e10
    if kind in ("resident", "whole") and (n > 200_000 or (nc == 1 and n > 12000)):
        return None
    p = _problem(case, seed)
    if kind == "precond":
        g = torch.Generator(device="cuda").manual_seed(seed + 5)
        return _precond(case, p, torch.randn(n, dtype=torch.float64, device="cuda", generator=g))
    if kind == "resident" and nc == 3:
        p["top_pressure"] = 1.0
    val, col, b, mask = _system(p)
    if kind == "spmv":
        g = torch.Generator(device="cuda").manual_seed(seed + 5)
        return _csr(val, col) @ torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    if kind == "assemble":
        return (None, None, val[col >= 0].reshape(-1), b)
    if kind == "resident":
        b = torch.where(mask, b, b + _load(case, p, seed))
    return _solve(val, col, b)
