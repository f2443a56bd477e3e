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
