"""The fused red-black kernel at the sides of the grid and of its tiles: every wall alone and all
together, whole and ragged tiles, grids narrower than a tile, one and two planes, each consumer
layout, against the oracle's solution (the bounds of the other FP32-inner solves)."""
import numpy as np
import pytest

import oracle
from paper_1410_1942_gb300 import build, capi, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available()
    build.build()
    capi.load()


@pytest.mark.parametrize("prec,tile", [("fp32", 31812108), ("fp32", 31812204), ("fp32", 33712204),
                                       ("fp32", 31712208), ("bf16", 31812108)])
@pytest.mark.parametrize("shape", [(64, 8, 5), (72, 17, 9), (136, 33, 7), (8, 3, 2), (16, 9, 1),
                                   (192, 32, 4)])
@pytest.mark.parametrize("walls", [0, 1, 2, 4, 8, 16, 31])
def test_solution_matches_the_oracle(walls, shape, prec, tile):
    nx, ny, nz = shape
    rng = np.random.default_rng(nx + ny + walls)
    F = rng.random((nz, ny, nx))
    F[rng.random(F.shape) < 0.3] = 0.0
    F[rng.random(F.shape) < 0.3] = 1.0
    h = 1.0 / nz
    s_ = rng.standard_normal(F.shape)
    op, b = oracle.operator(F, walls=walls), oracle.rhs(s_, h)
    with capi.Poisson(nx, ny, nz, h, precision=prec, precond="rbssor", tile=tile,
                      dirichlet_walls=walls) as s:
        assert "red-black" in s.describe()
        s.set_density(F)
        p = np.zeros(F.shape)
        rc, _ = s.solve(s_, p, 1e-9)
    assert rc == capi.OK
    assert oracle.rel_residual(op, b, p) <= 1e-9 * (1 + 1e-6)
    ref = oracle.pcg(op, b, tol=1e-12, precond="ssor").x
    assert np.linalg.norm(p - ref) <= 1e-6 * np.linalg.norm(ref)
