"""Projections in other units of length.

With the cell width times s, sbar over s and the velocity as it is, the right-hand
side is that of the unit box over s and phi that of the unit box times s.  For s a
power of two every operation of a solve scales without rounding, so the V-cycle
count is the same and phi equal bit for bit after division by s, unless some
intermediate leaves the range of its type.  Stars in centimetres have cells of
1e5 to 1e9; the boxes take every form of the bottom solve: one and two cells
(nodes) per thread, vectors in shared memory, vectors in global memory.
"""
import numpy as np
import pytest
import torch

from paper_1908_03634_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P, N, D = W.PERIODIC, W.NEUMANN, W.DIRICHLET
DEV = torch.device("cuda:0")
SCALES = [2.0**-20, 2.0**20, 2.0**33]


@pytest.fixture(scope="module")
def mx():
    from paper_1908_03634_gb300 import build as b
    b.build()
    import paper_1908_03634_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(mx):
    c = mx.mx_create(0)
    yield c
    mx.mx_destroy(c)


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def solve(mx, ctx, nodal, n, bc, s, **kw):
    g = W.Geom(tuple(n), s / n[0], tuple(bc), tuple(bc))
    rng = np.random.default_rng(5)
    cs = mx.cell_shape(g)
    # a contrast of 1e5 along z, as the stratified boxes have
    strat = 10.0 ** np.linspace(0.0, -5.0, n[2])[:, None, None]
    rho = cuda(np.exp(0.3 * rng.standard_normal(cs)) * strat)
    beta0 = cuda(np.ones(cs) * strat)
    sbar = cuda(rng.standard_normal(cs) / s)
    if nodal:
        u = [cuda(rng.standard_normal(cs)) for _ in range(3)]
        phi = torch.zeros(mx.node_shape(g), dtype=torch.float64, device=DEV)
        call = mx.mx_nodal_project
    else:
        u = [torch.from_numpy(rng.standard_normal(g.face_shape(d))) for d in range(3)]
        u = [t.to(DEV).contiguous() for t in W._periodic_faces(g, u)]
        phi = torch.zeros(cs, dtype=torch.float64, device=DEV)
        call = mx.mx_mac_project
    st, info = call(ctx, g, *u, rho, beta0, sbar, phi, mx.default_opts(**kw), allow=(mx.MX_OK, mx.MX_ERR_NOCONV))
    return info, phi / s


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("n,bc,kw", [((32, 32, 32), (P, P, N), {}), ((20, 24, 28), (P, P, N), {}),
                                     ((22, 26, 18), (N, D, N), {}), ((15, 13, 17), (D, N, D), {}),
                                     ((17, 17, 17), (D, N, N), {})])
def test_mac_in_other_units(mx, ctx, n, bc, kw, s):
    one, a = solve(mx, ctx, False, n, bc, 1.0, **kw)
    info, b = solve(mx, ctx, False, n, bc, s, **kw)
    assert one["status"] == 0 and one["rel_resid"] <= 1e-10
    assert (info["status"], info["vcycles"]) == (0, one["vcycles"])
    assert torch.equal(a, b)


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("n,bc", [((20, 24, 28), (P, P, N)), ((22, 26, 18), (N, D, N)), ((13, 13, 13), (D, N, N))])
def test_mac_fp64_in_other_units(mx, ctx, n, bc, s):
    test_mac_in_other_units(mx, ctx, n, bc, {"prec": 0}, s)


@pytest.mark.parametrize("s", SCALES)
def test_mac_fcg_in_other_units(mx, ctx, s):
    test_mac_in_other_units(mx, ctx, (20, 24, 28), (P, P, N), {"krylov": 1}, s)


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("n,bc,kw", [((24, 20, 28), (P, P, N), {}), ((12, 20, 28), (N, N, N), {"smoother": 1}),
                                     ((18, 14, 22), (N, N, N), {})])
def test_nodal_in_other_units(mx, ctx, n, bc, kw, s):
    one, a = solve(mx, ctx, True, n, bc, 1.0, **kw)
    info, b = solve(mx, ctx, True, n, bc, s, **kw)
    assert one["status"] == 0 and one["rel_resid"] <= 1e-10
    assert (info["status"], info["vcycles"]) == (0, one["vcycles"])
    assert torch.equal(a, b)


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("n,bc", [((24, 20, 28), (P, P, N)), ((18, 14, 22), (N, N, N))])
def test_nodal_fp64_in_other_units(mx, ctx, n, bc, s):
    test_nodal_in_other_units(mx, ctx, n, bc, {"prec": 0}, s)
