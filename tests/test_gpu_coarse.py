"""The coarse end of the MAC V-cycle (one launch over a thread-block cluster) at
the sizes where its layout changes: levels on one CTA or spread over 2 to 16,
slabs with and without a neighbour across a periodic z axis, an uneven last slab,
bottoms of one cell, one warp, several warps, two cells per thread, and more than
the register solve holds.

phi against the FP64 oracle solved to 1e-13 within the projection's 1e-8 bar, in
both precisions; and where the hierarchy ends in a level of at most 4096 cells,
the batched solve (one CTA per box, other cells per thread) bit for bit equal to
the single one.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1908_03634_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P, N, D = W.PERIODIC, W.NEUMANN, W.DIRICHLET
DEV = torch.device("cuda:0")

CASES = [
    ((2, 2, 2), (P, P, N)),       # the bottom alone, 8 cells
    ((4, 4, 4), (N, P, P)),       # one level above it, periodic z
    ((8, 12, 20), (P, D, N)),     # 1920 cells spread, bottom 2 x 3 x 5
    ((16, 16, 16), (P, P, P)),    # spread, periodic z: the last slab next to the first
    ((20, 24, 28), (P, P, N)),    # two spread levels, 14 slabs, bottom 5 x 6 x 7
    ((36, 44, 28), (D, D, D)),    # the finest level has its own kernels, bottom 9 x 11 x 7
    ((32, 32, 32), (N, N, P)),    # 16 slabs
    ((64, 16, 12), (P, P, N)),    # wide planes, 6 slabs of 8 CTAs
    ((22, 26, 18), (N, D, N)),    # bottom 11 x 13 x 9: 1287 cells, two per thread
    ((15, 13, 17), (D, N, D)),    # odd: bottom of 3315 cells, vectors in shared memory
]


@pytest.fixture(scope="module")
def mx():
    from paper_1908_03634_gb300 import build as b
    b.build()
    O.build()
    import paper_1908_03634_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(mx):
    c = mx.mx_create(0)
    yield c
    mx.mx_destroy(c)


def problem(n, bc, seed=5):
    g = W.Geom(tuple(n), 1.0 / n[0], tuple(bc), tuple(bc))
    rng = np.random.default_rng(seed)
    cs = O.cell_shape(g)
    rho, beta0 = np.exp(0.5 * rng.standard_normal(cs)), np.exp(0.5 * rng.standard_normal(cs))
    sbar = rng.standard_normal(cs)
    u = W._periodic_faces(g, [torch.from_numpy(rng.standard_normal(g.face_shape(d))) for d in range(3)])
    return g, rho, beta0, sbar, [t.numpy() for t in u]


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("n,bc", CASES)
def test_coarse_end_parity_and_batched_identity(mx, ctx, n, bc):
    g, rho, beta0, sbar, u = problem(n, bc)
    _, ref, info = O.mac_project(g, u, rho, beta0, sbar, tol=1e-13, maxit=400)
    assert info["ok"]
    phis = {}
    for prec in (0, 1):
        phi = torch.zeros(O.cell_shape(g), dtype=torch.float64, device=DEV)
        mx.mx_mac_project(ctx, g, *[cuda(t) for t in u], cuda(rho), cuda(beta0), cuda(sbar), phi,
                          mx.default_opts(prec=prec))
        phis[prec] = phi.cpu().numpy()
        assert np.abs(phis[prec] - ref).max() <= 1e-8 * np.abs(ref).max()
    phi = torch.zeros(O.cell_shape(g), dtype=torch.float64, device=DEV)
    mx.mx_mac_project_batched(ctx, [g], *[[cuda(t)] for t in u], [cuda(rho)], [cuda(beta0)], [cuda(sbar)], [phi],
                              mx.default_opts())
    assert np.array_equal(phi.cpu().numpy(), phis[1])


@pytest.mark.parametrize("n,bc", [((64, 64, 1), (P, P, N)), ((128, 32, 1), (D, N, N)), ((1, 4096, 1), (N, D, D)),
                                  ((5, 16, 32), (N, P, D)), ((13, 13, 15), (D, N, D))])
def test_largest_bottoms(mx, ctx, n, bc):
    """The largest bottoms the launch takes: 4096 cells in FP32 (one plane, one row), 2560
    in FP64, whose vectors fill the shared memory.  Batched solves take no box without a
    level that fits, so these calls fail where the layout leaves too little room.  The
    residual is the one asked for, 1e-10 of max |f|, up to the rounding of the row's twelve
    products (FP64; double-float coefficients in mixed solves), and the batched solve has the single one's bits."""
    g, rho, beta0, sbar, u = problem(n, bc)
    f, b = O.mac_rhs(g, u, beta0, sbar)[0], O.mac_coeffs(g, rho, beta0)
    phis = []
    for prec in (0, 1):
        phi = torch.zeros(O.cell_shape(g), dtype=torch.float64, device=DEV)
        mx.mx_mac_project(ctx, g, *[cuda(t) for t in u], cuda(rho), cuda(beta0), cuda(sbar), phi,
                          mx.default_opts(prec=prec))
        phis.append(phi.cpu().numpy())
        rounding = 2.0 ** (-44 if prec else -48) * 12 * max(np.abs(x).max() for x in b) * np.abs(phis[-1]).max() / g.dx**2
        assert np.abs(f - O.mac_apply(g, b, phis[-1])).max() <= 1e-10 * np.abs(f).max() + rounding
    phi = torch.zeros(O.cell_shape(g), dtype=torch.float64, device=DEV)
    mx.mx_mac_project_batched(ctx, [g], *[[cuda(t)] for t in u], [cuda(rho)], [cuda(beta0)], [cuda(sbar)], [phi],
                              mx.default_opts())
    assert np.array_equal(phi.cpu().numpy(), phis[1])


def flux(g, b, x):
    """sum over the faces of b times the neighbour's value (0 beyond a face without one)"""
    out = np.zeros_like(x)
    for d in range(3):
        ax = 2 - d
        n = x.shape[ax]
        lo, hi = np.roll(x, 1, ax), np.roll(x, -1, ax)
        if g.lo[d] != P:
            np.moveaxis(lo, ax, 0)[0] = 0.0
            np.moveaxis(hi, ax, 0)[-1] = 0.0
        out += np.take(b[d], range(n), ax) * lo + np.take(b[d], range(1, n + 1), ax) * hi
    return out


def diagonal(b):
    return sum(np.take(b[d], range(b[d].shape[2 - d] - 1), 2 - d) + np.take(b[d], range(1, b[d].shape[2 - d]), 2 - d)
               for d in range(3))


def vcycle(g, b, f, h, nu):
    """One V-cycle on L e = f in FP64 with an exact bottom solve, and the bound 1e-4 of
    the bottom residual's norm puts on the bottom's error."""
    n = f.shape
    den = diagonal(b)
    if any(k % 2 or k < 4 for k in n):
        m = np.empty((f.size, f.size))
        for c in range(f.size):
            unit = np.zeros(f.size)
            unit[c] = 1.0
            unit = unit.reshape(n)
            m[:, c] = (flux(g, b, unit) - den * unit).ravel() / h**2
        free = f - f.mean() if O.singular(g) else f
        s = np.linalg.svd(m, compute_uv=False)
        least = s[s > 1e-9 * s[0]].min()
        e = np.linalg.lstsq(m, free.ravel(), rcond=1e-9)[0].reshape(n)
        return e - (e.mean() if O.singular(g) else 0.0), 1e-4 * np.linalg.norm(free) / least
    colour = np.indices(n).sum(axis=0) % 2
    e = np.zeros(n)

    def smooth():
        for _ in range(nu):
            for c in (0, 1):
                e[colour == c] = ((flux(g, b, e) - h**2 * f) / den)[colour == c]

    smooth()
    r = f - (flux(g, b, e) - den * e) / h**2
    pairs = lambda a: a.reshape(n[0] // 2, 2, n[1] // 2, 2, n[2] // 2, 2)
    bc = [0.25 * sum(b[0][i::2, j::2, ::2] for i in (0, 1) for j in (0, 1)),
          0.25 * sum(b[1][i::2, ::2, j::2] for i in (0, 1) for j in (0, 1)),
          0.25 * sum(b[2][::2, i::2, j::2] for i in (0, 1) for j in (0, 1))]
    ec, bound = vcycle(g, bc, pairs(r).mean(axis=(1, 3, 5)), 2 * h, nu)
    pairs(e)[...] += ec[:, None, :, None, :, None]
    smooth()
    return e, bound


@pytest.mark.parametrize("n,bc", [((4, 4, 4), (N, P, P)), ((8, 12, 20), (P, D, N)), ((16, 16, 16), (P, P, P)),
                                  ((20, 24, 28), (P, P, N)), ((36, 28, 20), (D, D, D)), ((32, 32, 32), (N, N, P)),
                                  ((64, 16, 12), (P, P, N))])
@pytest.mark.parametrize("nu", [1, 2])
def test_one_fp64_vcycle(mx, ctx, n, bc, nu):
    """phi after one FP64 V-cycle against the same cycle in numpy with an exact bottom
    solve.  The bottom's error is at most 1e-4 of its right-hand side's norm over the
    least singular value; prolongation copies it and the smoother's rows are averages, so
    no value of phi is off by more, beyond rounding (1e-11 of max |phi|)."""
    g, rho, beta0, sbar, u = problem(n, bc)
    f, b = O.mac_rhs(g, u, beta0, sbar)[0], O.mac_coeffs(g, rho, beta0)
    for d in range(3):  # half a cell from the centre to a Dirichlet face
        for side, at in ((g.lo[d], 0), (g.hi[d], -1)):
            if side == D:
                np.moveaxis(b[d], 2 - d, 0)[at] *= 2.0
    want, bound = vcycle(g, b, f, g.dx, nu)
    want -= want.mean() if O.singular(g) else 0.0
    phi = torch.zeros(O.cell_shape(g), dtype=torch.float64, device=DEV)
    mx.mx_mac_project(ctx, g, *[cuda(t) for t in u], cuda(rho), cuda(beta0), cuda(sbar), phi,
                      mx.default_opts(prec=0, nu1=nu, nu2=nu, max_outer=1), allow=(mx.MX_OK, mx.MX_ERR_NOCONV))
    off = np.abs(phi.cpu().numpy() - want).max()
    assert bound <= 0.1 * np.abs(want).max()  # or the comparison would say little
    assert off <= (2 if O.singular(g) else 1) * bound + 1e-11 * np.abs(want).max()


@pytest.mark.parametrize("n", [(1, 1, 2), (3, 5, 7), (3, 5, 17), (9, 7, 15), (15, 13, 17), (17, 17, 17)])
@pytest.mark.parametrize("bc", [(N, N, N), (N, D, N)])
@pytest.mark.parametrize("prec", [0, 1])
def test_bottom_solve_alone(mx, ctx, n, bc, prec):
    """Boxes of one level: a V-cycle is the bottom solve, in each of its forms, to 1e-4 of
    the right-hand side's 2-norm, so at most 1e-4 sqrt(cells) of its maximum; the same
    again for the rounding of the iterates."""
    g, rho, beta0, sbar, u = problem(n, bc)
    phi = torch.zeros(O.cell_shape(g), dtype=torch.float64, device=DEV)
    st, info = mx.mx_mac_project(ctx, g, *[cuda(t) for t in u], cuda(rho), cuda(beta0), cuda(sbar), phi,
                                 mx.default_opts(prec=prec, max_outer=1), allow=(mx.MX_OK, mx.MX_ERR_NOCONV))
    assert info["vcycles"] <= 1 and info["rel_resid"] <= 2e-4 * np.sqrt(phi.numel())
