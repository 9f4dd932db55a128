"""Rows of any length on the one-sweep marching kernels (nx not a multiple of 8: the inner vectors
and rho/2 at a pitch), against the oracle and the column kernels.  Forced tiles take small grids
there; the default does for grids that do not fit on chip."""
import numpy as np
import pytest

import oracle
from paper_1410_1942_gb300 import build, capi, inputs

pytestmark = pytest.mark.gpu

L2_TOL = 1e-6


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available()
    build.build()
    capi.load()


def _solve(c, prec, tile, walls=0, tol=None, **kw):
    g = c.grid
    with capi.Poisson(g.nx, g.ny, g.nz, g.h, precision=prec, tile=tile, dirichlet_walls=walls,
                      **kw) as s:
        s.set_density(c.F)
        p = np.zeros(g.shape)
        rc, st = s.solve(c.s, p, tol or c.tol, allow=(capi.OK, capi.ENOTCONV))
        return rc, st, p, s.describe()


# one and two columns, one under and over a tile (64) and a row of eight, odd, even and prime
@pytest.mark.parametrize("tile", [10012204, 12012204, 13312204, 10312208])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("walls", [0, 31])
@pytest.mark.parametrize("shape", [(1, 9, 5), (2, 9, 5), (7, 20, 11), (9, 8, 9), (63, 17, 6),
                                   (65, 16, 7), (66, 9, 4), (101, 33, 12), (127, 24, 9)])
def test_solves_match_the_oracle(shape, walls, prec, tile):
    c = inputs.flat_case(*shape, seed=3, tol=1e-9)
    op, b = oracle.operator(c.F, walls=walls), oracle.rhs(c.s, c.grid.h)
    rc, st, p, desc = _solve(c, prec, tile, walls)
    assert rc == capi.OK and "march" in desc, desc
    rel = oracle.rel_residual(op, b, p)
    assert rel <= c.tol * (1 + 1e-6), rel
    ref = oracle.pcg(op, b, tol=1e-12, precond="ssor").x
    assert np.linalg.norm(p - ref) <= L2_TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("k", [7, 8])
def test_a_capped_solve_returns_the_k_th_iterate(k):
    c = inputs.strut_case(61, 24, 24, seed=2)
    op, b = oracle.operator(c.F), oracle.rhs(c.s, c.grid.h)
    rc, st, p, _ = _solve(c, "fp32", 12012204, max_iters=k)
    assert rc == capi.ENOTCONV and st["inner_iters"] == k
    ref = oracle.pcg(op, b, tol=0.0, precond="jacobi", max_iters=k).x
    assert np.linalg.norm(p - ref) <= 1e-4 * np.linalg.norm(ref)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_a_large_odd_grid_streams_by_default(prec):
    """The same pressure as the column kernels to the two residuals' tolerance (1e-11 each,
    amplified at most 100 times in the pressure of these cases: 2e-9), alone and in a batch with a
    grid of whole rows."""
    c = inputs.flat_case(187, 97, 90, seed=6, tol=1e-11)
    rc, _, q, _ = _solve(c, prec, -1)
    assert rc == capi.OK
    rc, _, p, desc = _solve(c, prec, 0)
    assert rc == capi.OK and "one-sweep" in desc and "march" in desc, desc
    assert np.linalg.norm(p - q) <= 2e-9 * np.linalg.norm(q)
    d = inputs.flat_case(192, 96, 90, seed=7, tol=1e-11)
    solvers, ps = [], []
    for x in (d, c):
        g = x.grid
        solvers.append(capi.Poisson(g.nx, g.ny, g.nz, g.h, precision=prec))
        solvers[-1].set_density(x.F)
        ps.append(np.zeros(g.shape))
    for t in capi.batch_submit(solvers, [d.s, c.s], ps, 1e-11):
        while True:
            rc, _ = capi.poll(t)
            if rc != capi.PENDING:
                break
        assert rc == capi.OK
    for s in solvers:
        s.close()
    assert np.linalg.norm(ps[1] - q) <= 2e-9 * np.linalg.norm(q)
    op, b = oracle.operator(d.F), oracle.rhs(d.s, d.grid.h)
    assert oracle.rel_residual(op, b, ps[0]) <= 1e-11 * (1 + 1e-6)


def test_apertures_move_the_handle_to_the_column_kernels_and_back():
    c = inputs.flat_case(45, 24, 20, seed=8, tol=1e-9)
    g = c.grid
    Lx, Ly, _ = g.lengths
    aps = inputs.cut_apertures(
        g, lambda x, y, z: inputs.ellipse_sdf(x, y, 0.5 * Lx, 0.5 * Ly, 0.3 * Lx, 0.2 * Ly))
    with capi.Poisson(g.nx, g.ny, g.nz, g.h, tile=12012204) as s:
        for a in (None, aps, None):
            s.set_apertures(*(a or ()))
            s.set_density(c.F)
            p = np.zeros(g.shape)
            rc, _ = s.solve(c.s, p, c.tol)
            assert rc == capi.OK
            op = oracle.operator(c.F, apertures=a) if a else oracle.operator(c.F)
            b = oracle.rhs(c.s, g.h, a[3]) if a else oracle.rhs(c.s, g.h)
            assert oracle.rel_residual(op, b, p) <= c.tol * (1 + 1e-6)
