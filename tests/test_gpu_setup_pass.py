"""The operator pass and the divisions of the projection passes, bit for bit against the oracle:
cells inside one phase, at interfaces and at boundaries, fractions that are only nearly 0 or 1,
and divisions over the whole exponent range."""
import numpy as np
import pytest

import oracle
from paper_1410_1942_gb300 import build, capi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    capi.load()


def _phases(shape, seed):
    """Water below air with a block of each in the other, and a few cells of other values."""
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    F = np.zeros(shape)
    F[: nz // 2] = 1.0
    F[nz // 4: nz // 4 + 2, ny // 3:, nx // 3:] = 0.0
    F[-3:-1, : ny // 2, : nx // 2] = 1.0
    odd = np.array([-0.0, 5e-324, 1e-300, 0.5, 1.0 - 2.0 ** -53, 1.0 + 2.0 ** -52, 0.25])
    at = rng.random(shape) < 0.02
    F[at] = rng.choice(odd, int(at.sum()))
    return F


@pytest.mark.parametrize("rho", [(1.0, 1000.0), (1.225, 998.2), (1000.0, 1.0), (3.0, 3.0)])
@pytest.mark.parametrize("nx,ny,nz,walls,per,cut", [
    (40, 24, 20, 0, False, False), (33, 17, 9, 31, False, False), (24, 16, 12, 20, True, False),
    (1, 9, 8, 3, False, False), (1, 6, 7, 0, True, False), (7, 1, 5, 8, False, False),
    (129, 3, 1, 0, False, False), (20, 12, 16, 2, False, True), (12, 10, 14, 4, True, True)])
def test_operator_bit_exact(nx, ny, nz, walls, per, cut, rho):
    shape = (nz, ny, nx)
    F = _phases(shape, nx + ny)
    aps = None
    if cut:
        rng = np.random.default_rng(3)
        aps = [rng.random(s) * (rng.random(s) < 0.9)
               for s in ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx), shape)]
        if per:
            aps[0][:, :, -1] = aps[0][:, :, 0]
    op = oracle.operator(F, *rho, walls=walls | (oracle.PERIODIC_X if per else 0), apertures=aps)
    for prec in ("fp64", "fp32"):
        with capi.Poisson(nx, ny, nz, 0.1, precision=prec, dirichlet_walls=walls,
                          periodic_x=per) as s:
            if cut:
                s.set_apertures(*aps)
            s.set_density(F, *rho)
            arrs = [np.empty(shape) for _ in range(4)]
            s.get_operator(*arrs)
        for got, ref in zip(arrs, (op.bx, op.by, op.bz, op.diag)):
            assert np.array_equal(got, ref)


@pytest.mark.parametrize("h,dt", [(1.0 / 3, 1.0), (0.1, 7e-5), (1.0, 1.0), (1e-3, 1.3e-3),
                                  (np.nextafter(2.0, 0), 1.0), (1e-200, 1.0), (1e180, 1.0)])
def test_division_over_the_exponent_range(h, dt):
    """One value to a cell (the z-velocity above it), its exponent from the subnormals up."""
    nx, ny, nz = 64, 32, 40
    rng = np.random.default_rng(5)
    u, v = np.zeros((nz, ny, nx + 1)), np.zeros((nz, ny + 1, nx))
    w = np.zeros((nz + 1, ny, nx))
    a = rng.uniform(1.0, 2.0, (nz // 2, ny, nx)) * rng.choice([-1.0, 1.0], (nz // 2, ny, nx))
    w[1::2] = np.ldexp(a, rng.integers(-1074, 1023, a.shape))
    w[1::2][rng.random(a.shape) < 0.05] = -0.0
    ref = oracle.divergence(u, v, w, h, dt)
    got = np.empty((nz, ny, nx))
    with capi.Poisson(nx, ny, nz, h) as s:
        s.divergence(u, v, w, dt, got)
    assert np.array_equal(got.view(np.int64), ref.view(np.int64))
