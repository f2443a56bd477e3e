"""The single-pass red-black sweep against the two colour passes at the edges of
its tiles: widths of exactly one tile, one column of pairs into the next and not
a multiple of four pairs; rows that fill the last tile, leave one row in it or
wrap; chunks of one plane run and of several; walls, Dirichlet and periodic faces
on every axis.  Both do per cell the same rounded operations, so after two
V-cycles phi is equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_1908_03634_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P, N, D = W.PERIODIC, W.NEUMANN, W.DIRICHLET
DEV = torch.device("cuda:0")


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


@pytest.mark.parametrize("n,bc", [((60, 112, 48), (P, P, N)), ((64, 98, 48), (D, D, D)), ((36, 128, 64), (P, D, P)),
                                  ((124, 30, 72), (D, P, D)), ((244, 16, 72), (N, N, P)), ((240, 140, 8), (P, N, D)),
                                  ((32, 16, 512), (D, N, N)), ((512, 4, 128), (N, P, D))])
@pytest.mark.parametrize("nu", [(1, 1), (2, 3)])
def test_sweep_bits(mx, ctx, n, bc, nu):
    g = W.Geom(n, 1.0 / n[0], bc, bc)
    rng = np.random.default_rng(2)
    cs = mx.cell_shape(g)
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    rho, beta0 = cuda(np.exp(0.5 * rng.standard_normal(cs))), cuda(np.exp(0.5 * rng.standard_normal(cs)))
    sbar = cuda(rng.standard_normal(cs))
    u = W._periodic_faces(g, [torch.from_numpy(rng.standard_normal(g.face_shape(d))) for d in range(3)])
    out = []
    for fused in (0, 1):
        phi = torch.zeros(cs, dtype=torch.float64, device=DEV)
        st, info = mx.mx_mac_project(ctx, g, *[cuda(t.numpy()) for t in u], rho, beta0, sbar, phi,
                                     mx.default_opts(fused=fused, nu1=nu[0], nu2=nu[1], max_outer=2),
                                     allow=(mx.MX_OK, mx.MX_ERR_NOCONV))
        assert info["vcycles"] == 2 and np.isfinite(info["rel_resid"])
        out.append(phi.cpu().numpy())
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("nu", [(1, 3), (2, 2)])
def test_batched_sweeps_equal_single_colour_passes(mx, ctx, nu):
    """A batch large enough for single-pass sweeps on its finest level (6 M cells)
    against single solves of its boxes, which run colour passes: the same bits."""
    boxes = [((128, 128, 128), (P, P, N)), ((160, 128, 144), (P, D, N)), ((64, 64, 64), (D, D, D)),
             ((128, 112, 136), (N, P, P))]
    rng = np.random.default_rng(4)
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    gs, rho, beta0, sbar, us = [], [], [], [], []
    for n, bc in boxes:
        g = W.Geom(n, 1.0 / n[0], bc, bc)
        cs = mx.cell_shape(g)
        gs.append(g)
        rho.append(cuda(np.exp(0.5 * rng.standard_normal(cs))))
        beta0.append(cuda(np.exp(0.5 * rng.standard_normal(cs))))
        sbar.append(cuda(rng.standard_normal(cs)))
        us.append(W._periodic_faces(g, [torch.from_numpy(rng.standard_normal(g.face_shape(d))) for d in range(3)]))
    assert sum(n[0] * n[1] * n[2] for n, _ in boxes) >= 6 << 20
    opts = mx.default_opts(nu1=nu[0], nu2=nu[1], max_outer=2)
    allow = (mx.MX_OK, mx.MX_ERR_NOCONV)
    phi = [torch.zeros_like(r) for r in rho]
    mx.mx_mac_project_batched(ctx, gs, *[[cuda(u[d].numpy()) for u in us] for d in range(3)], rho, beta0, sbar, phi,
                              opts, allow=allow)
    for b, g in enumerate(gs):
        one = torch.zeros_like(rho[b])
        mx.mx_mac_project(ctx, g, *[cuda(t.numpy()) for t in us[b]], rho[b], beta0[b], sbar[b], one, opts, allow=allow)
        assert torch.equal(one, phi[b])


def test_restriction_by_columns_equals_one_cell_per_thread(mx, ctx):
    """A batch of a million cells restricts by 2 x 2 columns per thread, single solves of
    its boxes by one cell per thread: the same bits.  Rows of one and two tiles of 64
    and a few pairs more, rows of blocks and chunks of planes that end early, every
    kind of face on every axis."""
    boxes = [((132, 24, 28), (D, P, N)), ((68, 36, 40), (P, N, D)), ((36, 132, 20), (N, D, P)),
             ((128, 8, 72), (P, P, P)), ((96, 96, 96), (P, P, N))]
    assert sum(n[0] * n[1] * n[2] for n, _ in boxes) >= 1 << 20 > max(n[0] * n[1] * n[2] for n, _ in boxes)
    rng = np.random.default_rng(6)
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    gs, rho, beta0, sbar, us = [], [], [], [], []
    for n, bc in boxes:
        g = W.Geom(n, 1.0 / n[0], bc, bc)
        cs = mx.cell_shape(g)
        gs.append(g)
        rho.append(cuda(np.exp(0.5 * rng.standard_normal(cs))))
        beta0.append(cuda(np.exp(0.5 * rng.standard_normal(cs))))
        sbar.append(cuda(rng.standard_normal(cs)))
        us.append(W._periodic_faces(g, [torch.from_numpy(rng.standard_normal(g.face_shape(d))) for d in range(3)]))
    opts = mx.default_opts(max_outer=2)
    allow = (mx.MX_OK, mx.MX_ERR_NOCONV)
    phi = [torch.zeros_like(r) for r in rho]
    mx.mx_mac_project_batched(ctx, gs, *[[cuda(u[d].numpy()) for u in us] for d in range(3)], rho, beta0, sbar, phi,
                              opts, allow=allow)
    for b, g in enumerate(gs):
        one = torch.zeros_like(rho[b])
        mx.mx_mac_project(ctx, g, *[cuda(t.numpy()) for t in us[b]], rho[b], beta0[b], sbar[b], one, opts, allow=allow)
        assert torch.equal(one, phi[b]), boxes[b]


def big_problem(mx, n, bc, seed):
    g = W.Geom(n, 1.0 / n[0], bc, bc)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rand = lambda s: torch.randn(s, dtype=torch.float64, device=DEV, generator=gen)
    cs = mx.cell_shape(g)
    rho, beta0 = torch.exp(0.5 * rand(cs)), torch.exp(0.5 * rand(cs))
    return g, rho, beta0, rand(cs), [t.contiguous() for t in W._periodic_faces(g, [rand(g.face_shape(d)) for d in range(3)])]


@pytest.mark.parametrize("n,bc", [((256, 256, 256), (P, P, N)), ((244, 200, 136), (D, P, N)), ((448, 126, 112), (N, D, P))])
@pytest.mark.parametrize("nu", [(2, 3), (1, 1)])
def test_sweeps_of_large_levels_equal_colour_passes(mx, ctx, n, bc, nu):
    """fused = 0 on levels of 6 M cells and more, where the sweep is the default, and
    fused = 1 on those below, against fused = 2: colour passes on every level."""
    g, rho, beta0, sbar, u = big_problem(mx, n, bc, 8)
    assert n[0] * n[1] * n[2] >= 6 << 20
    out = []
    for fused in (2, 0, 1):
        phi = torch.zeros_like(rho)
        st, info = mx.mx_mac_project(ctx, g, *[t.clone() for t in u], rho, beta0, sbar, phi,
                                     mx.default_opts(fused=fused, nu1=nu[0], nu2=nu[1], max_outer=2),
                                     allow=(mx.MX_OK, mx.MX_ERR_NOCONV))
        assert info["vcycles"] == 2 and np.isfinite(info["rel_resid"])
        out.append(phi)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
    mx.mx_profile_enable(ctx, True)
    for fused, launches in ((2, 2 * nu[0] + 1 + 2 * nu[1]), (0, nu[0] + nu[1])):
        mx.mx_profile_read(ctx)
        mx.mx_mac_project(ctx, g, *[t.clone() for t in u], rho, beta0, sbar, torch.zeros_like(rho),
                          mx.default_opts(fused=fused, nu1=nu[0], nu2=nu[1], max_outer=2), allow=(mx.MX_OK, mx.MX_ERR_NOCONV))
        assert mx.mx_profile_read(ctx)["smooth_fine"][1] == 2 * launches
    mx.mx_profile_enable(ctx, False)


def test_batched_and_composite_calls_take_the_option(mx, ctx):
    """The same bits from batches and composites whose levels sweep (fused = 1) and whose
    levels do not (2)."""
    boxes = [big_problem(mx, n, bc, 9) for n, bc in [((64, 48, 96), (P, P, N)), ((96, 40, 64), (D, N, P))]]
    allow = (mx.MX_OK, mx.MX_ERR_NOCONV)
    out = []
    for fused in (2, 1, 0):
        phi = [torch.zeros_like(b[1]) for b in boxes]
        mx.mx_mac_project_batched(ctx, [b[0] for b in boxes], *[[b[4][d].clone() for b in boxes] for d in range(3)],
                                  [b[1] for b in boxes], [b[2] for b in boxes], [b[3] for b in boxes], phi,
                                  mx.default_opts(fused=fused, max_outer=2), allow=allow)
        out.append(phi)
    assert all(torch.equal(a, b) and torch.equal(a, c) for a, b, c in zip(*out))
    coarse = big_problem(mx, (64, 64, 64), (P, P, N), 10)
    fine = big_problem(mx, (64, 64, 64), (N, N, N), 11)
    out = []
    for fused in (2, 1, 0):
        pc, pf = torch.zeros_like(coarse[1]), torch.zeros_like(fine[1])
        mx.mx_mac_project_composite(ctx, coarse[0], (16, 16, 16), (48, 48, 48), [t.clone() for t in coarse[4]], *coarse[1:4],
                                    pc, [t.clone() for t in fine[4]], *fine[1:4], pf,
                                    mx.default_opts(fused=fused, max_outer=2), allow=allow)
        out.append((pc, pf))
    assert all(torch.equal(out[0][k], out[m][k]) for k in (0, 1) for m in (1, 2))
