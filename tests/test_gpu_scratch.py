"""Loop graphs after the context's reduction scratch has moved.

A residual on a long thin box needs more partial results than a context starts
with, so the scratch is allocated anew; the plans of calls made before it keep
their loops as graphs.  Each kind of solve is repeated after that: the same bits as
before, and nothing written to memory that the library gave back (blocks of the
old scratch's size, taken from the driver in between, keep their pattern).
"""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1908_03634_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P, N, D = W.PERIODIC, W.NEUMANN, W.DIRICHLET
DEV = torch.device("cuda:0")
OLD_BYTES = 3 * 8 * (1 << 17)   # the scratch a context starts with
LONG = (1, 17, 350008)          # three blocks for every eight planes: 131253 partial results


@pytest.fixture(scope="module")
def mx():
    from paper_1908_03634_gb300 import build as b
    b.build()
    import paper_1908_03634_gb300 as m
    return m


class Blocks:
    """Device memory straight from the runtime, in blocks of the old scratch's size."""

    def __init__(self, count):
        self.rt = C.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
        self.ptr = []
        for _ in range(count):
            p = C.c_void_p()
            assert self.rt.cudaMalloc(C.byref(p), C.c_size_t(OLD_BYTES)) == 0
            assert self.rt.cudaMemset(p, C.c_int(0x5A), C.c_size_t(OLD_BYTES)) == 0
            self.ptr.append(p)

    def untouched(self):
        host = np.empty(OLD_BYTES, np.uint8)
        for p in self.ptr:
            assert self.rt.cudaMemcpy(C.c_void_p(host.ctypes.data), p, C.c_size_t(OLD_BYTES), C.c_int(2)) == 0
            if not (host == 0x5A).all():
                return False
        return True

    def free(self):
        for p in self.ptr:
            self.rt.cudaFree(p)


def rand(shape, rng):
    return torch.from_numpy(rng.standard_normal(shape)).to(DEV)


def solver(mx, ctx, kind):
    """A call of one kind on fixed inputs; returns its phi."""
    rng = np.random.default_rng(7)
    g = W.Geom((24, 16, 32), 1.0 / 24, (P, P, N), (P, P, N))
    cs = mx.cell_shape(g)
    rho, beta0 = torch.exp(0.5 * rand(cs, rng)), torch.exp(0.5 * rand(cs, rng))
    sbar = rand(cs, rng)
    faces = W._periodic_faces(g, [torch.from_numpy(rng.standard_normal(g.face_shape(d))) for d in range(3)])
    faces = [t.to(DEV).contiguous() for t in faces]
    cells = [rand(cs, rng) for _ in range(3)]

    def call():
        nodal = kind.startswith("nodal")
        u = [t.clone() for t in (cells if nodal else faces)]
        phi = torch.zeros(mx.node_shape(g) if nodal else cs, dtype=torch.float64, device=DEV)
        o = mx.default_opts(prec=0 if kind.endswith("fp64") else 1)
        if nodal:
            mx.mx_nodal_project(ctx, g, *u, rho, beta0, sbar, phi, o)
        elif kind == "batched":
            mx.mx_mac_project_batched(ctx, [g, g], *[[t, t.clone()] for t in u], [rho] * 2, [beta0] * 2, [sbar] * 2,
                                      [phi, phi.clone()], o)
        else:
            mx.mx_mac_project(ctx, g, *u, rho, beta0, sbar, phi, o)
        return phi

    return call


@pytest.mark.parametrize("kind", ["mac", "mac_fp64", "batched", "nodal", "nodal_fp64"])
def test_solves_after_the_scratch_has_moved(mx, kind):
    ctx = mx.mx_create(0)
    blocks = None
    try:
        call = solver(mx, ctx, kind)
        before = call()
        g = W.Geom(LONG, 1.0, (N, N, N), (N, N, N))
        one = torch.ones(mx.cell_shape(g), dtype=torch.float64, device=DEV)
        r = torch.empty_like(one)
        mx.mx_residual(ctx, g, mx.MX_OP_MAC, 0, one, one, one, one, r)
        assert torch.equal(r, one)  # L of a constant is 0 between walls
        blocks = Blocks(16)
        after = call()
        torch.cuda.synchronize()
        assert torch.equal(before, after)
        assert blocks.untouched()
    finally:
        if blocks:
            blocks.free()
        mx.mx_destroy(ctx)
