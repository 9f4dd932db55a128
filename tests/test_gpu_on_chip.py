"""Jacobi-PCG held on chip (grids that fit the registers and shared memory of the GPU): every
operator form, box edges of one cell, odd sizes, the largest grids that fit, and the launch's own
bookkeeping, against the oracle and against the column kernels (tile -1)."""
import numpy as np
import pytest

import oracle
from paper_1410_1942_gb300 import build, capi, inputs

pytestmark = pytest.mark.gpu

L2_TOL = 1e-6
PERIODIC = oracle.PERIODIC_X


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available()
    build.build()
    capi.load()


def _solve(c, tol, prec, tile=0, walls=0, aps=None, **kw):
    g = c.grid
    with capi.Poisson(g.nx, g.ny, g.nz, g.h, precision=prec, tile=tile,
                      dirichlet_walls=walls & 31, periodic_x=bool(walls & PERIODIC), **kw) as s:
        if aps is not None:
            s.set_apertures(*aps)
        s.set_density(c.F)
        p = np.zeros(g.shape)
        rc, st = s.solve(c.s, p, tol, allow=(capi.OK, capi.ENOTCONV))
        return rc, st, p, s.describe()


def _check(c, op, b, p, tol):
    rel = oracle.rel_residual(op, b, p)
    assert rel <= tol * (1 + 1e-6), rel
    ref = oracle.pcg(op, b, tol=1e-12, precond="ssor").x
    assert np.linalg.norm(p - ref) <= L2_TOL * np.linalg.norm(ref)


# one cell, lines, planes, one box exactly, one cell over a box, odd sizes, thin and long
SHAPES = [(1, 1, 1), (5, 1, 1), (1, 7, 3), (2, 2, 2), (32, 16, 16), (33, 17, 17), (37, 23, 19),
          (64, 48, 32), (7, 90, 20), (150, 5, 3), (31, 33, 50)]


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("shape", SHAPES)
def test_solves_match_the_oracle(shape, prec):
    c = inputs.flat_case(*shape, seed=3, tol=1e-9)
    op, b = oracle.operator(c.F), oracle.rhs(c.s, c.grid.h)
    rc, st, p, desc = _solve(c, c.tol, prec)
    assert rc == capi.OK and "on chip" in desc, desc
    _check(c, op, b, p, c.tol)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("walls", [31, 2 | 8, PERIODIC, PERIODIC | 4 | 16])
@pytest.mark.parametrize("shape", [(2, 3, 4), (40, 24, 20), (70, 33, 18)])
def test_walls_and_wrap_match_the_oracle(shape, walls, prec):
    c = inputs.flat_case(*shape, seed=4, tol=1e-9)
    op, b = oracle.operator(c.F, walls=walls), oracle.rhs(c.s, c.grid.h)
    rc, st, p, desc = _solve(c, c.tol, prec, walls=walls)
    assert rc == capi.OK and "on chip" in desc, desc
    _check(c, op, b, p, c.tol)


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
def test_cut_cells_match_the_oracle(prec):
    c = inputs.flat_case(50, 33, 26, seed=5, tol=1e-9)
    Lx, Ly, _ = c.grid.lengths
    aps = inputs.cut_apertures(
        c.grid, lambda x, y, z: inputs.ellipse_sdf(x, y, 0.5 * Lx, 0.5 * Ly, 0.3 * Lx, 0.2 * Ly))
    op = oracle.operator(c.F, apertures=aps)
    b = oracle.rhs(c.s, c.grid.h, aps[3])
    rc, st, p, desc = _solve(c, c.tol, prec, aps=aps)
    assert rc == capi.OK and "cut-cells" in desc and "on chip" in desc, desc
    _check(c, op, b, p, c.tol)
    assert not np.any(p[aps[3] == 0])


@pytest.mark.parametrize("prec,shape", [("fp32", (160, 96, 80)), ("fp64", (128, 64, 64)),
                                        ("fp32", (161, 96, 80))])
def test_the_largest_grids_agree_with_the_column_kernels(prec, shape):
    """The largest grids on chip and one plane of columns more (which streams): the same pressure
    as the column kernels to the two residuals' tolerance (1e-11 each, amplified at most 100
    times in the pressure of these cases: 2e-9)."""
    c = inputs.flat_case(*shape, seed=6, tol=1e-11)
    rc, st, p, desc = _solve(c, c.tol, prec)
    assert rc == capi.OK and ("on chip" in desc) == (shape[0] != 161), desc
    rc, _, q, _ = _solve(c, c.tol, prec, tile=-1)
    assert rc == capi.OK and np.linalg.norm(p - q) <= 2e-9 * np.linalg.norm(q)


@pytest.mark.parametrize("prec,bound", [("fp32", 1e-4), ("fp64", 1e-9)])
@pytest.mark.parametrize("k", [1, 2, 7, 8])
def test_a_capped_solve_returns_the_k_th_iterate(prec, bound, k):
    """The k-th iterate of the oracle's textbook Jacobi PCG, in the arithmetic's accuracy."""
    c = inputs.strut_case(48, 24, 24, seed=2)
    op, b = oracle.operator(c.F), oracle.rhs(c.s, c.grid.h)
    rc, st, p, _ = _solve(c, 1e-9, prec, max_iters=k)
    assert rc == capi.ENOTCONV and st["inner_iters"] == k
    ref = oracle.pcg(op, b, tol=0.0, precond="jacobi", max_iters=k).x
    assert np.linalg.norm(p - ref) <= bound * np.linalg.norm(ref)


def test_tags_start_over_when_they_run_out():
    """Iteration caps of 2e9 use half of the 32-bit tags per inner solve: repeated solves clear the
    words and start over, with the same result every time."""
    c = inputs.flat_case(40, 24, 20, seed=7, tol=1e-9)
    g = c.grid
    with capi.Poisson(g.nx, g.ny, g.nz, g.h, max_iters=2_000_000_000) as s:
        s.set_density(c.F)
        out = []
        for _ in range(3):
            p = np.zeros(g.shape)
            rc, _ = s.solve(c.s, p, c.tol)
            assert rc == capi.OK
            out.append(p)
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


def test_small_and_large_sources_scale():
    """The inner solve's sums are taken on a residual scaled to norm one: sources 1e-15 and 1e15
    times as large give the scaled pressure (powers of two: bit for bit)."""
    c = inputs.flat_case(33, 17, 17, seed=8, tol=1e-9)
    ref = _solve(c, c.tol, "fp32")[2]
    for e in (-50, 50):
        d = inputs.Case(c.name, c.grid, c.F, np.ldexp(c.s, e), c.tol, c.meta)
        rc, _, p, _ = _solve(d, c.tol, "fp32")
        assert rc == capi.OK and np.array_equal(np.ldexp(p, -e), ref)


def test_an_unreachable_box_times_out_and_the_handle_recovers():
    c = inputs.strut_case(64, 32, 32, seed=2)
    g = c.grid
    with capi.Poisson(g.nx, g.ny, g.nz, g.h) as s:
        s.set_density(c.F)
        assert "on chip" in s.describe()
        s.test_unreachable_barrier(1)
        p = np.zeros(g.shape)
        rc, _ = s.solve(c.s, p, c.tol, allow=(capi.ETIMEOUT,))
        assert rc == capi.ETIMEOUT and np.all(np.isfinite(p))
        s.test_unreachable_barrier(0)
        p = np.zeros(g.shape)
        rc, _ = s.solve(c.s, p, c.tol)
        assert rc == capi.OK
    _check(c, oracle.operator(c.F), oracle.rhs(c.s, g.h), p, c.tol)


def test_a_batch_of_grids_on_chip_and_streamed_matches_each_alone():
    """Many small grids (more boxes than SMs: the CTAs run several solves one after another), odd
    and periodic ones, and one too large for the chip, in one batch."""
    shapes = [(160, 96, 96), (64, 48, 32), (37, 23, 19), (96, 64, 64), (32, 16, 16), (5, 1, 1)] + \
             [(64 + 8 * i, 48, 40 + i) for i in range(24)]
    cases = [inputs.flat_case(*s, seed=10 + i, tol=1e-9) for i, s in enumerate(shapes)]
    solvers, alone = [], []
    for i, c in enumerate(cases):
        g = c.grid
        s = capi.Poisson(g.nx, g.ny, g.nz, g.h, periodic_x=(i % 5 == 2))
        s.set_density(c.F)
        p = np.zeros(g.shape)
        assert s.solve(c.s, p, c.tol)[0] == capi.OK
        solvers.append(s)
        alone.append(p)
    ps = [np.zeros(c.grid.shape) for c in cases]
    for t in capi.batch_submit(solvers, [c.s for c in cases], ps, 1e-9):
        while True:
            rc, _ = capi.poll(t)
            if rc != capi.PENDING:
                break
        assert rc == capi.OK
    for s in solvers:
        s.close()
    for p, q in zip(ps, alone):
        assert np.linalg.norm(p - q) <= 2e-6 * np.linalg.norm(q)
