"""The V-cycle's fine passes on TMA-staged planes and the bottom levels in shared memory: ragged
tiles in x and y, odd rows and planes, a single plane, walls, BF16 densities, and the levels each
form of the bottom takes, against the oracle's cycle (bounds as in the V-cycle parity tests: FP64 sums
in another order, FP32 rounding through some forty sweeps and sums)."""
import numpy as np
import pytest

import oracle
from oracle import multigrid as mg
from paper_1410_1942_gb300 import build, capi, inputs

pytestmark = pytest.mark.gpu

VCYCLE_TOL = {"fp64": 1e-12, "fp32": 2e-5}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available()
    build.build()
    capi.load()


def _F(shape, seed):
    rng = np.random.default_rng(seed)
    F = rng.random(shape)
    F[rng.random(shape) < 0.3] = 0.0
    F[rng.random(shape) < 0.3] = 1.0
    return F


# one tile and less, one cell over a tile in y, whole and ragged tiles in x, odd ny and nz, one and
# two planes, chunks of several planes
SHAPES = [(8, 2, 1), (8, 3, 2), (64, 16, 2), (72, 17, 5), (136, 33, 7), (200, 15, 9), (56, 48, 67)]


@pytest.mark.parametrize("walls", [0, 1 | 8, 31])
@pytest.mark.parametrize("shape", SHAPES)
def test_vcycle_matches_the_oracle(shape, walls):
    nx, ny, nz = shape
    F = _F((nz, ny, nx), 1)
    r = np.random.default_rng(2).standard_normal((nz, ny, nx))
    want = mg.vcycle(mg.hierarchy(oracle.operator(F, walls=walls)), r)
    with capi.Poisson(nx, ny, nz, 1.0 / nz, precond="mg", dirichlet_walls=walls) as s:
        s.set_density(F)
        got = np.empty_like(r)
        s.precond_apply(r, got, kind="mg", precision="fp32")
    assert np.linalg.norm(got - want) <= VCYCLE_TOL["fp32"] * np.linalg.norm(want)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("walls", [0, 31])
@pytest.mark.parametrize("shape", [(72, 17, 21), (136, 40, 24)])
def test_solves_match_the_oracle(shape, walls, prec):
    c = inputs.flat_case(*shape, seed=3, tol=1e-9)
    g = c.grid
    op, b = oracle.operator(c.F, walls=walls), oracle.rhs(c.s, g.h)
    with capi.Poisson(g.nx, g.ny, g.nz, g.h, precision=prec, precond="mg", inner_tol=1e-5,
                      dirichlet_walls=walls) as s:
        s.set_density(c.F)
        for _ in range(2):  # the second through the captured chunk from its first iteration
            p = np.zeros(g.shape)
            rc, _ = s.solve(c.s, p, c.tol)
            assert rc == capi.OK
            assert oracle.rel_residual(op, b, p) <= c.tol * (1 + 1e-6)
    ref = oracle.pcg(op, b, tol=1e-12, precond="ssor").x
    assert np.linalg.norm(p - ref) <= 1e-6 * np.linalg.norm(ref)


# bottoms: one level only, 2048 cells and one more plane, several levels of a long line, a coarsest
# level of 512 cells, and (periodic, odd) one too large for shared memory
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shape,walls", [((16, 8, 8), 0), ((32, 32, 16), 0), ((32, 32, 17), 31),
                                         ((3000, 1, 1), 0), ((16, 16, 16), oracle.PERIODIC_X),
                                         ((2501, 2, 1), oracle.PERIODIC_X)])
def test_bottom_levels_match_the_oracle(shape, walls, prec):
    nx, ny, nz = shape
    F = _F((nz, ny, nx), 5)
    r = np.random.default_rng(6).standard_normal((nz, ny, nx))
    want = mg.vcycle(mg.hierarchy(oracle.operator(F, walls=walls)), r)
    with capi.Poisson(nx, ny, nz, 1.0 / nz, precision=prec, precond="mg",
                      dirichlet_walls=walls & 31, periodic_x=bool(walls & oracle.PERIODIC_X)) as s:
        s.set_density(F)
        got = np.empty_like(r)
        s.precond_apply(r, got, kind="mg", precision=prec)
    assert np.linalg.norm(got - want) <= VCYCLE_TOL[prec] * np.linalg.norm(want)


@pytest.mark.parametrize("periodic", [False, True])
def test_densities_whose_diagonal_has_a_flushed_reciprocal(periodic):
    """Diagonals of 1.3 * 2^126, whose FP32 reciprocal is below the normal numbers: the damped-Jacobi
    updates divide by them all the same.  p scales with the density."""
    shape = (1, 2, 64)
    rho = 6 / (2.0 ** 126 * 1.3)
    F = np.zeros(shape)
    b = np.random.default_rng(1).standard_normal(shape) * 1e10
    out = []
    for r in (1.0, rho):
        with capi.Poisson(64, 2, 1, 0.1, precond="mg", periodic_x=periodic, max_iters=300) as s:
            s.set_density(F, r, r)
            p = np.zeros(shape)
            rc, _ = s.solve(b, p, 1e-9, allow=(capi.OK, capi.ENOTCONV))
            assert rc == capi.OK, r
            out.append(p / r)
    assert np.linalg.norm(out[1] - out[0]) <= 1e-6 * np.linalg.norm(out[0])
