"""What is timed: the calls a low Mach number time step makes of this library.

Each case is one call, or one short run of calls, through the Python binding on
fields in device memory.  The workloads are the repository's own recipes
(`paper_1908_03634_gb300/workloads.py`): a planar stratified box (periodic in x
and y, walls in z, density contrast up to 1e5), the full star (Dirichlet faces,
contrast 1e6), patches of an adaptive grid, and the base-state mapping of the
star.  Fields follow the same formulas, drawn on the device so that the 512^3
inputs take a fraction of a second.

Extents are those geometric multigrid is used with: a small base extent (2 to
11 cells) times a power of two, different per axis in the ragged cases.  Solves
run to the relative residual of 1e-10 that the library's defaults ask for.
"""
import math

import torch

import paper_1908_03634_gb300 as mx

PERIODIC, NEUMANN, DIRICHLET = mx.MX_BC_PERIODIC, mx.MX_BC_NEUMANN, mx.MX_BC_DIRICHLET
DEV = "cuda"
F64 = torch.float64


class Geom:
    """Cell counts, cell width and the boundary type per axis."""

    def __init__(self, n, dx, bc):
        self.n, self.dx, self.lo, self.hi = tuple(n), dx, tuple(bc), tuple(bc)


# ---- the cases -------------------------------------------------------------------------


def _mac(name, n, field="planar", prec="mixed", nu1=2, nu2=2, krylov=0):
    c = {"kind": "mac", "nx": n[0], "ny": n[1], "nz": n[2], "field": field, "prec": prec, "nu1": nu1, "nu2": nu2,
         "krylov": krylov}
    return dict(c, name=name) if name else c


def _nodal(name, n, smoother=0, nu1=2, nu2=2):
    c = {"kind": "nodal", "nx": n[0], "ny": n[1], "nz": n[2], "smoother": smoother, "nu1": nu1, "nu2": nu2}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest whole projection, plain FP64 on the 32^3 smoke box: launches and latency count
        _mac("mac_planar32_fp64", (32, 32, 32), prec="fp64"),
        # one patch of an adaptive grid solved alone, ragged extents, the library's default options
        _mac("mac_patch_72x88x56", (72, 88, 56)),
        # the headline: planar 256^3, mixed precision, with the sweep counts the autotuner picks there
        _mac("mac_planar256", (256, 256, 256), nu1=2, nu2=3),
        # the full star, the largest MAC grid (Dirichlet faces), same sweeps
        _mac("mac_star512", (512, 512, 512), field="star", nu1=2, nu2=3),
        # the plain FP64 solve that the mixed one is held against, at an ordinary size
        _mac("mac_planar128_fp64", (128, 128, 128), prec="fp64"),
        # flexible CG around cheap V-cycles on a box that is not a cube
        _mac("mac_fcg_160x192x224", (160, 192, 224), nu1=1, nu2=2, krylov=1),
        # the nodal projection at its full size with the smoother the autotuner picks (Chebyshev)
        _nodal("nodal384_cheb", (384, 384, 384), smoother=1),
        # a ragged nodal box with the default smoother (four-colour Gauss-Seidel)
        _nodal("nodal_gs_96x80x112", (96, 80, 112)),
        # 96 uneven patches in one batched call
        {"name": "batched96", "kind": "batched", "npatch": 96, "largest": 128, "sizes_seed": 3, "nu1": 1, "nu2": 3},
        # two AMR levels: a coarse box and a patch of its own size around the heating
        {"name": "composite128", "kind": "composite", "n": 128, "p0": 32, "p1": 96, "field": "planar"},
        # lateral Average of the full star's density and the Fill back onto the cells
        {"name": "average_fill512", "kind": "average", "n": 512, "offset": 0},
        # velocity split of the star: w0 from the base state, w0 e_r on the faces, S - Sbar on the cells
        {"name": "split256", "kind": "split", "n": 256, "nr": 1024},
    ]


def _extents(rng, lo, hi, most):
    """Three extents in [lo, hi], each a base of 2 to 11 cells times one power of two, at most `most` cells."""
    while True:
        edge = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        k = max(2, int(math.log2(edge / rng.uniform(2.5, 9.0))))
        n = [min(11, max(2, round(edge * rng.uniform(0.7, 1.4) / 2 ** k))) << k for _ in range(3)]
        if all(lo <= v <= hi for v in n) and n[0] * n[1] * n[2] <= most:
            return n


def draw(rng):
    kind = rng.choice(["mac", "mac", "mac", "mac_fp64", "nodal", "nodal", "batched", "composite", "average", "split"])
    if kind == "mac":
        n = _extents(rng, 32, 448, 320 ** 3)
        krylov = int(rng.random() < 0.2)
        nu1, nu2 = rng.choice([(2, 2), (2, 2), (2, 3), (3, 3)] + ([(1, 2)] if krylov else []))
        field = rng.choice(["planar", "planar", "star"])
        if field == "star":
            n = [n[0]] * 3 if n[0] ** 3 <= 320 ** 3 else [256] * 3
        return _mac(None, n, field, "mixed", nu1, nu2, krylov)
    if kind == "mac_fp64":
        return _mac(None, _extents(rng, 32, 192, 160 ** 3), "planar", "fp64", *rng.choice([(2, 2), (2, 3)]))
    if kind == "nodal":
        n = _extents(rng, 32, 352, 288 ** 3)
        smoother = rng.randrange(2)
        nu1, nu2 = rng.choice([(2, 2), (1, 3), (2, 3)] if smoother else [(2, 2), (3, 3)])
        return _nodal(None, n, smoother, nu1, nu2)
    if kind == "batched":
        return {"kind": "batched", "npatch": round(math.exp(rng.uniform(math.log(4), math.log(96)))),
                "largest": rng.choice([64, 96, 128]), "sizes_seed": rng.randrange(1 << 20),
                "nu1": rng.choice([1, 2]), "nu2": rng.choice([2, 3])}
    if kind == "composite":
        n = rng.choice([48, 64, 80, 96, 112, 128])
        if rng.random() < 0.5:  # the star with a patch over its core
            p0 = rng.choice([n // 4, 3 * n // 8]) // 2 * 2
            return {"kind": "composite", "n": n, "p0": p0, "p1": n - p0, "field": "star"}
        p0 = rng.randrange(2, n // 8) * 2
        return {"kind": "composite", "n": n, "p0": p0, "p1": p0 + 8 * rng.randrange(2, (n - 2 - p0) // 8 + 1),
                "field": "planar"}
    if kind == "average":
        return {"kind": "average", "n": round(math.exp(rng.uniform(math.log(64), math.log(480)))),
                "offset": rng.choice([0, 0, 1, 7])}
    return {"kind": "split", "n": round(math.exp(rng.uniform(math.log(64), math.log(256)))),
            "nr": rng.randrange(200, 2048)}


def work(case):
    """Inputs read once and outputs written once; the flops of one operator application or sum over the fields."""
    kind = case["kind"]
    if kind in ("mac", "nodal"):  # U in and out, rho, beta0, Sbar in, phi out
        cells = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 80 * cells, "flops": (60 if kind == "mac" else 150) * cells}
    if kind == "batched":
        cells = sum(e ** 3 for e in _batch_edges(case))
        return {"bytes": 80 * cells, "flops": 60 * cells}
    if kind == "composite":
        cells = case["n"] ** 3 + (2 * (case["p1"] - case["p0"])) ** 3
        return {"bytes": 80 * cells, "flops": 60 * cells}
    cells = case["n"] ** 3
    if kind == "average":  # the field in, the filled field out
        return {"bytes": 16 * cells, "flops": cells}
    return {"bytes": 64 * cells, "flops": 7 * cells}  # three face arrays in and out, S in, S - Sbar out


# ---- fields ----------------------------------------------------------------------------

def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * seed + stream)


def _host_gen(seed, stream):
    return torch.Generator().manual_seed(1_000_003 * seed + stream)


def _centres(n, h, start=0.0):
    return start + (torch.arange(n, dtype=F64, device=DEV) + 0.5) * h


def _edges(n, h, start=0.0):
    return start + torch.arange(n + 1, dtype=F64, device=DEV) * h


def _points(n, h, d, start=(0.0, 0.0, 0.0)):
    """x, y, z coordinates of the d-face centres (d None: cell centres)."""
    return [(_edges if a == d else _centres)(n[a], h, start[a]) for a in range(3)]


def _modes(seed, m):
    """m Fourier modes: wavevectors in {-4..4}^3 without 0, phases, unit polarisations."""
    g = _host_gen(seed, 1)
    k = torch.randint(-4, 5, (m, 3), generator=g)
    k[(k == 0).all(1)] = torch.tensor([1, -2, 3])
    e = torch.randn((m, 3), generator=g, dtype=F64)
    phase = 2 * math.pi * torch.rand(m, generator=g, dtype=F64)
    return k.to(F64).to(DEV), phase.to(DEV), (e / e.norm(dim=1, keepdim=True)).to(DEV)


def _velocity(modes, comp, pts):
    """sum over modes of e[comp] sin(2 pi k.x + phase) on the grid of pts."""
    k, phase, e = modes
    w = [torch.exp(2j * math.pi * k[:, a, None] * pts[a][None, :]) for a in range(3)]
    wz = (e[:, comp, None] * torch.exp(1j * phase)[:, None]) * w[2]
    zy = (wz[:, :, None] * w[1][:, None, :]).reshape(k.shape[0], -1)
    nz, ny, nx = (len(pts[a]) for a in (2, 1, 0))
    return (zy.imag.T @ w[0].real + zy.real.T @ w[0].imag).reshape(nz, ny, nx)


def _hotspots(spots, pts):
    out = 0.0
    for c in spots:
        gx, gy, gz = (torch.exp(-((pts[a] - c[a]) ** 2) / 0.05 ** 2) for a in range(3))
        out = out + gz[:, None, None] * (gy[:, None] * gx[None, :])[None]
    return out


def _radius(pts):
    x, y, z = pts
    return torch.sqrt((z[:, None, None] - 0.5) ** 2 + (y[None, :, None] - 0.5) ** 2 + (x[None, None, :] - 0.5) ** 2)


def _star_rho0(r):
    return torch.where(r <= 0.45, (1.0 + (r / 0.05) ** 2) ** -2.5, torch.full_like(r, 1e-6))


def _wrap(u, bc):
    """On a periodic axis face n is the image of face 0."""
    for d in range(3):
        if bc[d] == PERIODIC:
            u[d].narrow(2 - d, u[d].shape[2 - d] - 1, 1).copy_(u[d].narrow(2 - d, 0, 1))
    return u


def _cell_fields(field, pts, seed, stream, contrast=1e5, height=1.0):
    """rho and beta0 at the cell centres pts; planar: rho0 falls by `contrast` over `height`."""
    shape = tuple(len(pts[a]) for a in (2, 1, 0))
    if field == "star":
        rho0 = _star_rho0(_radius(pts))
        beta0 = rho0 ** 0.6
    else:
        rho0 = torch.exp(-math.log(contrast) / height * pts[2])[:, None, None]
        beta0 = (rho0 ** 0.6).expand(shape).contiguous()
    xi = torch.rand(shape, generator=_gen(seed, stream), dtype=F64, device=DEV).mul_(0.02).add_(0.99)
    return xi.mul_(rho0), beta0


def _spots(field, seed, count=3):
    if field == "star":
        return [(0.5, 0.5, 0.5)]
    return (0.2 + 0.6 * torch.rand((count, 3), generator=_host_gen(seed, 2), dtype=F64)).tolist()


def _box(n, field, seed, modes, staggered=True, contrast=1e5, spots=3):
    """One projection problem: (geom, rho, beta0, sbar, [ux, uy, uz])."""
    h = 1.0 / n[0]
    bc = (DIRICHLET,) * 3 if field == "star" else (PERIODIC, PERIODIC, NEUMANN)
    cells = _points(n, h, None)
    rho, beta0 = _cell_fields(field, cells, seed, 3, contrast, n[2] * h)
    m = _modes(seed, modes)
    u = [_velocity(m, d, _points(n, h, d) if staggered else cells) for d in range(3)]
    if staggered:
        u = _wrap(u, bc)
    return Geom(n, h, bc), rho, beta0, _hotspots(_spots(field, seed, spots), cells), u


def _batch_edges(case):
    g = torch.Generator().manual_seed(case["sizes_seed"])
    sizes = [s for s in (32, 48, 64, 96, 128) if s <= case["largest"]]
    return [sizes[i] for i in torch.randint(0, len(sizes), (case["npatch"],), generator=g).tolist()]


# ---- what a program holds, and its pass ------------------------------------------------

_ctx = None


def _context():
    """The one library context of a program."""
    global _ctx
    if _ctx is None:
        _ctx = mx.mx_create(0)
    return _ctx


def _extent(case):
    return (case["nx"], case["ny"], case["nz"])


def _solve_box(case, seed):
    if case["kind"] == "mac":
        return _box(_extent(case), case["field"], seed, 32 if case["field"] == "star" else 16)
    return _box(_extent(case), "planar", seed, 16, staggered=False)


def _batch_boxes(case, seed):
    g = _host_gen(seed, 5)
    out = []
    for p, e in enumerate(_batch_edges(case)):
        contrast = 10.0 ** (2.0 + 3.0 * torch.rand(1, generator=g, dtype=F64).item())
        out.append(_box((e, e, e), "planar", 1000 * seed + p, 8, contrast=contrast, spots=1))
    return out


def _arena(fields):
    """A batch's fields in one allocation, each on a 512-byte boundary: the flat tensor and the fields in it."""
    at, total = [], 0
    for t in fields:
        at.append(total)
        total += -(-t.numel() // 64) * 64
    flat = torch.zeros(total, dtype=F64, device=DEV)
    views = [flat[a:a + t.numel()].view(t.shape) for a, t in zip(at, fields)]
    torch._foreach_copy_(views, list(fields))
    return flat, views


def _levels(case, seed):
    """Both levels of a composite problem: (geom, plo, phi, coarse fields, fine fields), fields (rho, beta0, sbar, u)."""
    n, plo, phi, field = case["n"], (case["p0"],) * 3, (case["p1"],) * 3, case["field"]
    H = 1.0 / n
    bc = (DIRICHLET,) * 3 if field == "star" else (PERIODIC, PERIODIC, NEUMANN)
    m, spots = _modes(seed, 8), [(0.5, 0.5, 0.5)]

    def level(counts, h, start, stream):
        cells = _points(counts, h, None, start)
        rho, beta0 = _cell_fields(field, cells, seed, stream)
        return rho, beta0, _hotspots(spots, cells), [_velocity(m, d, _points(counts, h, d, start)) for d in range(3)]

    coarse = level((n,) * 3, H, (0.0,) * 3, 3)
    _wrap(coarse[3], bc)
    fine = level([2 * (phi[a] - plo[a]) for a in range(3)], H / 2, [plo[a] * H for a in range(3)], 4)
    return Geom((n,) * 3, H, bc), plo, phi, coarse, fine


def _opts(case):
    o = mx.default_opts(nu1=case["nu1"], nu2=case["nu2"])
    o.prec = mx.MX_PREC_FP64 if case.get("prec") == "fp64" else mx.MX_PREC_MIXED
    o.krylov, o.smoother = case.get("krylov", 0), case.get("smoother", 0)
    return o


def _star_corner(n, offset):
    """The star's centre on a cell corner: the middle of the box, or some cells off it."""
    return (n // 2 + offset, n // 2, n // 2 - offset)


def _base_state(case, seed):
    """Base-state edges, beta0 and the w0 source on nr radial cells reaching past the box's corners."""
    nr = case["nr"]
    r_edge = torch.linspace(0.0, 0.9, nr + 1, dtype=F64, device=DEV)
    mid = 0.5 * (r_edge[1:] + r_edge[:-1])
    src = torch.exp(-(mid / 0.1) ** 2) * (1.0 + 0.1 * torch.rand(nr, generator=_gen(seed, 6), dtype=F64, device=DEV))
    return r_edge, _star_rho0(mid) ** 0.6, src


def _split_fields(case, seed):
    """Face velocities of the star and its constraint S: the central heating on a fluctuating background."""
    n = (case["n"],) * 3
    cells = _points(n, 1.0 / n[0], None)
    m = _modes(seed, 16)
    u = [_velocity(m, d, _points(n, 1.0 / n[0], d)) for d in range(3)]
    S = _hotspots([(0.5, 0.5, 0.5)], cells)
    S += 1e-3 * torch.rand(S.shape, generator=_gen(seed, 7), dtype=F64, device=DEV)
    return Geom(n, 1.0 / n[0], (DIRICHLET,) * 3), u, S


def _star_density(case, seed):
    n = (case["n"],) * 3
    return _cell_fields("star", _points(n, 1.0 / n[0], None), seed, 3)[0]


def prepare(case, seed):
    kind, s = case["kind"], {"case": case, "ctx": _context()}
    if kind in ("mac", "nodal"):
        s["geom"], s["rho"], s["beta0"], s["sbar"], s["u_adv"] = _solve_box(case, seed)
        shape = mx.cell_shape(s["geom"]) if kind == "mac" else mx.node_shape(s["geom"])
        s.update(opts=_opts(case), phi=torch.zeros(shape, dtype=F64, device=DEV),
                 u=[torch.empty_like(t) for t in s["u_adv"]])
    elif kind == "batched":
        boxes = _batch_boxes(case, seed)
        s["geoms"], s["rho"], s["beta0"], s["sbar"] = ([b[i] for b in boxes] for i in range(4))
        s["u_adv"] = [_arena([b[4][d] for b in boxes])[0] for d in range(3)]
        s["u"], s["views"] = zip(*(_arena([b[4][d] for b in boxes]) for d in range(3)))
        s["phi"], s["phi_views"] = _arena([torch.zeros_like(r) for r in s["rho"]])
        s["opts"] = _opts(case)
    elif kind == "composite":
        s["geom"], s["plo"], s["phi_hi"], s["coarse"], s["fine"] = _levels(case, seed)
        s["u_adv"] = s["coarse"][3] + s["fine"][3]
        s["u"] = [torch.empty_like(t) for t in s["u_adv"]]
        s["phi"] = [torch.zeros_like(s[level][0]) for level in ("coarse", "fine")]
    elif kind == "average":
        n = case["n"]
        s["geom"], s["corner"] = Geom((n,) * 3, 1.0 / n, (DIRICHLET,) * 3), _star_corner(n, case["offset"])
        s["rho"] = _star_density(case, seed)
        nb = mx.mx_radial_nbins(s["geom"], s["corner"])
        s.update(avg=torch.empty(nb, dtype=F64, device=DEV), count=torch.empty(nb, dtype=torch.int64, device=DEV),
                 out=torch.empty_like(s["rho"]))
    else:
        s["geom"], s["u_adv"], s["S"] = _split_fields(case, seed)
        s["r_edge"], s["beta0"], s["src"] = _base_state(case, seed)
        s.update(corner=_star_corner(case["n"], 0), w0=torch.empty_like(s["r_edge"]), out=torch.empty_like(s["S"]),
                 u=[torch.empty_like(t) for t in s["u_adv"]])
    return s


def run(s):
    kind, ctx = s["case"]["kind"], s["ctx"]
    if "u" in s:  # the advective velocity of this step; the projection overwrites it
        torch._foreach_copy_(list(s["u"]), s["u_adv"])
        u = s["u"]
    if kind == "mac":
        mx.mx_mac_project(ctx, s["geom"], *u, s["rho"], s["beta0"], s["sbar"], s["phi"], s["opts"])
        return [s["phi"]] + u
    if kind == "nodal":
        mx.mx_nodal_project(ctx, s["geom"], *u, s["rho"], s["beta0"], s["sbar"], s["phi"], s["opts"])
        return [s["phi"]] + u
    if kind == "batched":
        mx.mx_mac_project_batched(ctx, s["geoms"], *s["views"], s["rho"], s["beta0"], s["sbar"], s["phi_views"],
                                  s["opts"])
        return [s["phi"], *u]
    if kind == "composite":
        (rho_c, beta0_c, sbar_c, _), (rho_f, beta0_f, sbar_f, _) = s["coarse"], s["fine"]
        mx.mx_mac_project_composite(ctx, s["geom"], s["plo"], s["phi_hi"], u[:3], rho_c, beta0_c, sbar_c, s["phi"][0],
                                    u[3:], rho_f, beta0_f, sbar_f, s["phi"][1])
        return s["phi"] + u
    if kind == "average":
        mx.mx_average_radial(ctx, s["geom"], s["corner"], s["rho"], s["avg"], s["count"])
        mx.mx_fill_radial(ctx, s["geom"], s["corner"], s["avg"], s["out"])
        return [s["avg"], s["count"], s["out"]]
    mx.mx_w0_integrate(ctx, 1, s["r_edge"], s["beta0"], s["src"], s["w0"])
    mx.mx_add_w0_faces(ctx, s["geom"], 1, s["corner"], s["r_edge"], s["w0"], *u)
    mx.mx_subtract_lateral_average(ctx, s["geom"], 1, s["corner"], s["S"], s["out"])
    return [s["w0"], s["out"]] + u


# ---- the same results in 64 bits, in plain torch ---------------------------------------


def exact(case, seed):
    kind = case["kind"]
    if kind == "mac":
        return _exact_mac(*_solve_box(case, seed))
    if kind == "nodal":
        return _exact_nodal(*_solve_box(case, seed))
    if kind == "batched":
        solved = [_exact_mac(*box) for box in _batch_boxes(case, seed)]
        return [_arena([out[i] for out in solved])[0] for i in range(4)]
    if kind == "composite":
        return _exact_composite(*_levels(case, seed))
    if kind == "average":
        return _exact_average(case, seed)
    return _exact_split(case, seed)


def _pcg(apply, precondition, f, tol, most):
    """Preconditioned conjugate gradients for A x = f, A positive (semi)definite."""
    x, r = torch.zeros_like(f), f.clone()
    z = precondition(r)
    p, rz = z, (r * z).sum()
    stop = tol * f.abs().max().item()
    for _ in range(most):
        if r.abs().max().item() <= stop:
            break
        q = apply(p)
        a = rz / (p * q).sum()
        x.add_(p * a)
        r.sub_(q * a)
        z = precondition(r)
        rz, old = (r * z).sum(), rz
        p = z + p * (rz / old)
    return x


def _refined(apply, precondition, f, clean, tol=2e-12):
    """A x = f by restarted conjugate gradients on the recomputed residual; `clean` takes rounding out of the null space."""
    x, r, top = torch.zeros_like(f), f, f.abs().max().item()
    left = top
    for _ in range(6):
        if left <= tol * top:
            break
        y = clean(x + _pcg(apply, precondition, r, 1e-6, 100))
        ry = f - apply(y)
        now = ry.abs().max().item()
        if not now < 0.5 * left:  # rounding: no nearer
            break
        x, r, left = y, ry, now
    return x


def _eigen_1d(n, bc, nodal):
    """Eigenvectors and eigenvalues of minus the second difference on one axis (unit width; nodal: linear elements)."""
    m = n + 1 if nodal and bc != PERIODIC else n
    K, M = torch.zeros((m, m), dtype=F64), torch.eye(m, dtype=F64)
    i = torch.arange(m - 1)
    K[i, i] += 1.0
    K[i + 1, i + 1] += 1.0
    K[i, i + 1] -= 1.0
    K[i + 1, i] -= 1.0
    if bc == PERIODIC:
        for a, b, v in ((0, 0, 1.0), (m - 1, m - 1, 1.0), (0, m - 1, -1.0), (m - 1, 0, -1.0)):
            K[a, b] += v
    elif bc == DIRICHLET:
        K[0, 0] += 2.0
        K[m - 1, m - 1] += 2.0
    if nodal:
        M = torch.diag(torch.diagonal(K)) / 2.0 - K / 6.0  # lumped less K/6: the consistent mass
    K, M = K.to(DEV), M.to(DEV)
    L = torch.linalg.cholesky(M)
    A = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, K, upper=False).T, upper=False)
    lam, Q = torch.linalg.eigh(0.5 * (A + A.T))
    return lam, torch.linalg.solve_triangular(L.T, Q, upper=True)


def _separable(geom, scale, nodal=False):
    """r -> s^-1/2 (constant-coefficient solve) s^-1/2 r in FP32, s = scale: a good preconditioner for div(s grad)."""
    V, lam = [], []
    for a in range(3):
        w, Q = _eigen_1d(geom.n[a], geom.lo[a], nodal)
        V.append(Q.to(torch.float32))
        lam.append(w / geom.dx ** 2)
    inv = (1.0 / (lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :] + 5.0)).to(torch.float32)
    root = scale.rsqrt().to(torch.float32)

    def solve(r):
        top = r.abs().max().clamp_min(1e-300)
        t = (r / top).to(torch.float32) * root
        nz, ny, nx = t.shape
        t = torch.matmul(V[1].T, torch.matmul(t, V[0]))
        t = torch.matmul(V[2].T, t.reshape(nz, -1)).reshape(nz, ny, nx) * inv
        t = torch.matmul(V[2], t.reshape(nz, -1)).reshape(nz, ny, nx)
        t = torch.matmul(V[1], torch.matmul(t, V[0].T)) * root
        return t.to(F64) * top

    return solve


def _cut(t, d, a, b):
    """t[a:b] along axis d (x, y, z = 0, 1, 2)."""
    return t.narrow(2 - d, a, b - a)


def _face_values(c, d, bc):
    """Arithmetic means of the cell field on the d-faces; the cell's own value on a boundary face."""
    n = c.shape[2 - d]
    lo, hi = _cut(c, d, 0, 1), _cut(c, d, n - 1, n)
    if bc == PERIODIC:
        lo = hi = 0.5 * (lo + hi)
    return torch.cat([lo, 0.5 * (_cut(c, d, 0, n - 1) + _cut(c, d, 1, n)), hi], 2 - d)


def _face_gradient(phi, d, bc, h):
    """dphi/dn on the d-faces: 0 on walls, towards phi = 0 half a cell away on Dirichlet faces."""
    n = phi.shape[2 - d]
    lo, hi = _cut(phi, d, 0, 1), _cut(phi, d, n - 1, n)
    if bc == PERIODIC:
        first = last = lo - hi
    elif bc == DIRICHLET:
        first, last = 2.0 * lo, -2.0 * hi
    else:
        first, last = torch.zeros_like(lo), torch.zeros_like(hi)
    return torch.cat([first, _cut(phi, d, 1, n) - _cut(phi, d, 0, n - 1), last], 2 - d).div_(h)


def _divergence(flux, h):
    out = 0.0
    for d in range(3):
        n = flux[d].shape[2 - d]
        out = out + (_cut(flux[d], d, 1, n) - _cut(flux[d], d, 0, n - 1))
    return out / h


def _walls_closed(u, geom):
    """U with 0 on wall faces."""
    out = []
    for d in range(3):
        t = u[d].clone()
        if geom.lo[d] == NEUMANN:
            n = t.shape[2 - d]
            _cut(t, d, 0, 1).zero_()
            _cut(t, d, n - 1, n).zero_()
        out.append(t)
    return out


def _exact_mac(geom, rho, beta0, sbar, u):
    h, bc = geom.dx, geom.lo
    rho_f = [_face_values(rho, d, bc[d]) for d in range(3)]
    beta_f = [_face_values(beta0, d, bc[d]) for d in range(3)]
    b = [beta_f[d] / rho_f[d] for d in range(3)]
    u = _walls_closed(u, geom)
    f = beta0 * sbar - _divergence([beta_f[d] * u[d] for d in range(3)], h)  # minus the right-hand side
    singular = DIRICHLET not in bc
    clean = (lambda t: t - t.mean()) if singular else (lambda t: t)
    f = clean(f)

    def apply(phi):  # minus L: positive
        return -_divergence([b[d] * _face_gradient(phi, d, bc[d], h) for d in range(3)], h)

    phi = _refined(apply, _separable(geom, beta0 / rho), f, clean)
    return [phi] + [u[d] - _face_gradient(phi, d, bc[d], h) / rho_f[d] for d in range(3)]


def _corners(phi, geom):
    """The eight corner values of every cell, [z][y][x] offsets."""
    for d in range(3):
        if geom.lo[d] == PERIODIC:
            phi = torch.cat([phi, _cut(phi, d, 0, 1)], 2 - d)
    nx, ny, nz = geom.n
    return [[[phi[k:k + nz, j:j + ny, i:i + nx] for i in (0, 1)] for j in (0, 1)] for k in (0, 1)]


def _to_nodes(parts, geom):
    """Sum cell-corner contributions parts[k][j][i] onto the nodes."""
    nx, ny, nz = geom.n
    out = torch.zeros((nz + 1, ny + 1, nx + 1), dtype=F64, device=DEV)
    for k in (0, 1):
        for j in (0, 1):
            for i in (0, 1):
                out[k:k + nz, j:j + ny, i:i + nx] += parts(k, j, i)
    for d in range(3):
        if geom.lo[d] == PERIODIC:
            _cut(out, d, 0, 1).add_(_cut(out, d, geom.n[d], geom.n[d] + 1))
            out = _cut(out, d, 0, geom.n[d]).contiguous()
    return out


def _exact_nodal(geom, rho, beta0, sbar, u):
    h, sigma = geom.dx, beta0 / rho
    w = _to_nodes(lambda k, j, i: 1.0, geom) / 8.0
    bu = [beta0 * t for t in u]
    bs = beta0 * sbar

    def rhs_part(k, j, i):  # the node is the cell's corner (i, j, k): the cell lies on its + side where the index is 0
        s = (1 - 2 * i) * bu[0] + (1 - 2 * j) * bu[1] + (1 - 2 * k) * bu[2]
        return s / (4.0 * h) - bs / 8.0

    f = _to_nodes(rhs_part, geom)  # w times the right-hand side
    mean = f.sum() / w.sum()
    f = -(f - w * mean)

    def apply(phi):  # minus w L, positive semidefinite
        c = _corners(phi, geom)
        tetra = [sum(c[k][j][i] for k in (0, 1) for j in (0, 1) for i in (0, 1) if (i + j + k) % 2 == p)
                 for p in (0, 1)]

        def part(k, j, i):
            y = tetra[(i + j + k) % 2] - 5.0 * c[k][j][i] + c[1 - k][1 - j][1 - i]
            return y.mul_(sigma).mul_(-1.0 / (12.0 * h * h))

        return _to_nodes(part, geom)

    scale = _to_nodes(lambda k, j, i: sigma, geom) / (8.0 * w)
    total = w.sum()
    phi = _refined(apply, _separable(geom, scale, nodal=True), f, lambda t: t - (w * t).sum() / total)
    c = _corners(phi, geom)
    grad = [sum((1 if (i, j, k)[d] else -1) * c[k][j][i] for k in (0, 1) for j in (0, 1) for i in (0, 1)) / (4.0 * h)
            for d in range(3)]
    return [phi] + [u[d] - grad[d] / rho for d in range(3)]


def _children(t):
    """Means over 2 x 2 x 2 blocks."""
    nz, ny, nx = t.shape
    return t.reshape(nz // 2, 2, ny // 2, 2, nx // 2, 2).mean((1, 3, 5))


def _face_means(t, d):
    """Means of the fine d-faces over the four on each coarse d-face (even face planes)."""
    t = t.index_select(2 - d, torch.arange(0, t.shape[2 - d], 2, device=DEV))
    for a in range(3):
        if a != d:
            t = 0.5 * (t.index_select(2 - a, torch.arange(0, t.shape[2 - a], 2, device=DEV))
                       + t.index_select(2 - a, torch.arange(1, t.shape[2 - a], 2, device=DEV)))
    return t


def _doubled(t, d):
    """A plane of coarse values repeated on the fine tangential positions."""
    for a in range(3):
        if a != d:
            t = t.repeat_interleave(2, 2 - a)
    return t


class _Composite:
    """The two-level operator: fine ghosts by linear tangential and quadratic normal interpolation, coarse fluxes on
    the interface the means of the fine ones."""

    def __init__(self, geom, plo, phi, coarse, fine):
        self.g, self.plo, self.phi, self.bc = geom, plo, phi, geom.lo
        self.H, self.h = geom.dx, geom.dx / 2
        self.box = tuple(slice(plo[a], phi[a]) for a in (2, 1, 0))
        cf = []
        for c, f in zip(coarse[:2], fine[:2]):  # face values of rho and beta0 on both levels
            fc = [_face_values(c, d, self.bc[d]) for d in range(3)]
            ff = []
            for d in range(3):
                t = _face_values(f, d, NEUMANN)
                m = t.shape[2 - d]
                _cut(t, d, 0, 1).copy_(0.5 * (_cut(f, d, 0, 1) + _doubled(self.across(c, d, -1), d)))
                _cut(t, d, m - 1, m).copy_(0.5 * (_cut(f, d, m - 2, m - 1) + _doubled(self.across(c, d, 1), d)))
                ff.append(t)
            cf.append((fc, ff))
        (self.rho_c, self.rho_f), (self.beta_c, self.beta_f) = cf
        self.b_c = [self.beta_c[d] / self.rho_c[d] for d in range(3)]
        self.b_f = [self.beta_f[d] / self.rho_f[d] for d in range(3)]

    def across(self, c, d, side, shift=(0, 0, 0)):
        """The plane of coarse cells across the patch face along d, moved by `shift` cells."""
        at = [slice(self.plo[a] + shift[a], self.phi[a] + shift[a]) for a in range(3)]
        q = self.plo[d] - 1 if side < 0 else self.phi[d]
        at[d] = slice(q, q + 1)
        return c[at[2], at[1], at[0]]

    def ghost(self, pc, pf, d, side):
        m = pf.shape[2 - d]
        f1, f2 = (_cut(pf, d, 0, 1), _cut(pf, d, 1, 2)) if side < 0 else (_cut(pf, d, m - 1, m), _cut(pf, d, m - 2, m - 1))
        c = _doubled(self.across(pc, d, side), d)
        for a in range(3):
            if a != d:
                e = tuple(int(x == a) for x in range(3))
                slope = _doubled(self.across(pc, d, side, e) - self.across(pc, d, side, tuple(-x for x in e)), d) / 8.0
                sign = torch.ones(slope.shape[2 - a], dtype=F64, device=DEV)
                sign[0::2] = -1.0
                shape = [1, 1, 1]
                shape[2 - a] = -1
                c = c + slope * sign.reshape(shape)
        return 8.0 / 15.0 * c + 2.0 / 3.0 * f1 - 0.2 * f2

    def gradients(self, pc, pf):
        gc = [_face_gradient(pc, d, self.bc[d], self.H) for d in range(3)]
        gf = []
        for d in range(3):
            t = _face_gradient(pf, d, NEUMANN, self.h)
            m = t.shape[2 - d]
            _cut(t, d, 0, 1).copy_((_cut(pf, d, 0, 1) - self.ghost(pc, pf, d, -1)) / self.h)
            _cut(t, d, m - 1, m).copy_((self.ghost(pc, pf, d, 1) - _cut(pf, d, m - 2, m - 1)) / self.h)
            gf.append(t)
        return gc, gf

    def matched(self, fc, ff):
        """Coarse faces on and inside the patch take the means of the fine faces."""
        for d in range(3):
            at = [slice(self.plo[a], self.phi[a] + (1 if a == d else 0)) for a in range(3)]
            fc[d][at[2], at[1], at[0]] = _face_means(ff[d], d)
        return fc

    def divergence(self, fc, ff):
        dc = _divergence(self.matched(fc, ff), self.H)
        dc[self.box] = 0.0
        return dc, _divergence(ff, self.h)

    def apply(self, pc, pf):
        gc, gf = self.gradients(pc, pf)
        return self.divergence([self.b_c[d] * gc[d] for d in range(3)], [self.b_f[d] * gf[d] for d in range(3)])

    def mean(self, c, f):
        cells = c.numel() - f.numel() // 8
        c = c.clone()
        c[self.box] = 0.0
        return ((c.sum() + f.sum() / 8) / (cells + f.numel() / 8)).item()


def _exact_composite(geom, plo, phi, coarse, fine):
    G = _Composite(geom, plo, phi, coarse, fine)
    uc, uf = _walls_closed(coarse[3], geom), [t.clone() for t in fine[3]]
    dc, df = G.divergence([G.beta_c[d] * uc[d] for d in range(3)], [G.beta_f[d] * uf[d] for d in range(3)])
    fc, ff = dc - coarse[1] * coarse[2], df - fine[1] * fine[2]
    singular = DIRICHLET not in geom.lo
    if singular:
        m = G.mean(fc, ff)
        fc, ff = fc - m, ff - m
    fc[G.box] = 0.0
    top = max(fc.abs().max().item(), ff.abs().max().item())

    # corrections by level: the whole coarse box, then the patch with its ghosts' share of the diagonal
    b = [t.clone() for t in G.b_c]
    G.matched(b, G.b_f)
    rho_c, beta_c = coarse[0].clone(), coarse[1].clone()
    rho_c[G.box], beta_c[G.box] = _children(fine[0]), _children(fine[1])
    bf = [t.clone() for t in G.b_f]
    for d in range(3):
        n = bf[d].shape[2 - d]
        for a in (0, n - 1):
            _cut(bf[d], d, a, a + 1).mul_(4.0 / 15.0)  # 8/15 b where a Dirichlet face has 2 b
    patch = Geom(tuple(fine[0].shape[2 - a] for a in range(3)), G.h, (DIRICHLET,) * 3)
    pre_c, pre_f = _separable(geom, beta_c / rho_c), _separable(patch, fine[1] / fine[0])

    def minus_l(coef, bc, h):
        return lambda p: -_divergence([coef[d] * _face_gradient(p, d, bc[d], h) for d in range(3)], h)

    a_c, a_f = minus_l(b, geom.lo, G.H), minus_l(bf, patch.lo, G.h)
    pc, pf = torch.zeros_like(fc), torch.zeros_like(ff)
    rc, rf, best = fc, ff, math.inf
    for _ in range(60):
        now = max(rc.abs().max().item(), rf.abs().max().item())
        if now <= 1e-14 * top or (now < 1e-12 * top and now > 0.7 * best):
            break
        best = min(best, now)
        r = rc.clone()
        r[G.box] = _children(rf)
        if singular:
            r = r - r.mean()
        ec = _pcg(a_c, pre_c, -r, 1e-3, 200)
        pc = pc + ec
        pf = pf + ec[G.box].repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)
        _, lf = G.apply(pc, pf)
        pf = pf + _pcg(a_f, pre_f, lf - ff, 1e-3, 200)
        lc, lf = G.apply(pc, pf)
        rc, rf = fc - lc, ff - lf
        rc[G.box] = 0.0
    if singular:
        m = G.mean(pc, pf)
        pc, pf = pc - m, pf - m
    gc, gf = G.gradients(pc, pf)
    uc = [uc[d] - gc[d] / G.rho_c[d] for d in range(3)]
    uf = [uf[d] - gf[d] / G.rho_f[d] for d in range(3)]
    G.matched(uc, uf)
    pc[G.box] = _children(pf)
    return [pc, pf] + uc + uf


def _bins(n, corner):
    """Radial bin of every cell: T(a) + T(b) + T(c), T(a) = a (a + 1) / 2, of its distances to the corner."""
    t = []
    for d in range(3):
        a = torch.arange(n, device=DEV, dtype=torch.int64) - corner[d]
        t.append(a * (a + 1) // 2)
    return t[2][:, None, None] + t[1][None, :, None] + t[0][None, None, :]


def _bin_means(field, bins, nb):
    flat = bins.reshape(-1)
    count = torch.bincount(flat, minlength=nb)
    total = torch.zeros(nb, dtype=F64, device=DEV).index_add_(0, flat, field.reshape(-1))
    return total / count.clamp_min(1), count


def _exact_average(case, seed):
    n = case["n"]
    bins = _bins(n, _star_corner(n, case["offset"]))
    nb = int(bins.max().item()) + 1
    avg, count = _bin_means(_star_density(case, seed), bins, nb)
    return [avg, count, avg[bins]]


def _exact_split(case, seed):
    geom, u, S = _split_fields(case, seed)
    r_edge, beta0, src = _base_state(case, seed)
    n, corner = case["n"], _star_corner(case["n"], 0)
    q = torch.cat([torch.zeros(1, dtype=F64, device=DEV),
                   torch.cumsum((r_edge[1:] ** 3 - r_edge[:-1] ** 3) / 3.0 * beta0 * src, 0)])
    edge = torch.cat([beta0[:1], 0.5 * (beta0[1:] + beta0[:-1]), beta0[-1:]])
    w0 = torch.where(r_edge > 0, q / (r_edge ** 2 * edge).clamp_min(1e-300), torch.zeros_like(q))
    bins = _bins(n, corner)
    mean, _ = _bin_means(S, bins, int(bins.max().item()) + 1)
    out = [w0, S - mean[bins]]
    centre = [corner[a] * geom.dx for a in range(3)]
    for d in range(3):
        p = _points(geom.n, geom.dx, d)
        x = [p[a] - centre[a] for a in range(3)]
        r = torch.sqrt(x[2][:, None, None] ** 2 + x[1][None, :, None] ** 2 + x[0][None, None, :] ** 2)
        j = (torch.searchsorted(r_edge, r.reshape(-1), right=True) - 1).clamp(0, len(r_edge) - 2).reshape(r.shape)
        t = (r - r_edge[j]) / (r_edge[j + 1] - r_edge[j])
        w = torch.where(r >= r_edge[-1], w0[-1] * (r_edge[-1] / r) ** 2, (1.0 - t) * w0[j] + t * w0[j + 1])
        shape = [1, 1, 1]
        shape[2 - d] = -1
        out.append(u[d] + w * x[d].reshape(shape) / r.clamp_min(1e-300))
    return out
