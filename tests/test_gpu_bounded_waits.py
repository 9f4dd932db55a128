"""The bounded waits of the on-chip PCG and of the V-cycle's fine passes: a wait that runs out ends the
solve with ETIMEOUT (nothing faults or hangs), and the same handle then solves as if nothing had
happened."""
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


def _check(op, b, p, tol):
    rel = oracle.rel_residual(op, b, p)
    assert rel <= tol * (1 + 1e-6), rel
    ref = oracle.pcg(op, b, tol=1e-12, precond="ssor").x
    assert np.linalg.norm(p - ref) <= L2_TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("prec,cut", [("fp64", False), ("fp64", True), ("fp32", True),
                                      ("bf16", False)])
def test_an_unreachable_box_times_out_in_every_precision(prec, cut):
    c = inputs.strut_case(64, 32, 32, seed=2)
    g = c.grid
    aps = None
    if cut:
        Lx, Ly, _ = g.lengths
        aps = inputs.cut_apertures(
            g, lambda x, y, z: inputs.ellipse_sdf(x, y, 0.5 * Lx, 0.5 * Ly, 0.3 * Lx, 0.2 * Ly))
    with capi.Poisson(g.nx, g.ny, g.nz, g.h, precision=prec) as s:
        if cut:
            s.set_apertures(*aps)
        s.set_density(c.F)
        assert "on chip" in s.describe(), s.describe()
        s.test_unreachable_box(1)
        p = np.zeros(g.shape)
        rc, _ = s.solve(c.s, p, c.tol, allow=(capi.ETIMEOUT,))
        assert rc == capi.ETIMEOUT and np.all(np.isfinite(p))
        s.test_unreachable_box(0)
        p = np.zeros(g.shape)
        rc, _ = s.solve(c.s, p, c.tol)
        assert rc == capi.OK
    if cut:
        _check(oracle.operator(c.F, apertures=aps), oracle.rhs(c.s, g.h, aps[3]), p, c.tol)
    else:
        _check(oracle.operator(c.F), oracle.rhs(c.s, g.h), p, c.tol)


def test_a_box_that_waits_for_a_long_solve_before_it_is_no_timeout():
    """One solve on nearly every SM with ten times the iterations its grid suggests, and small solves
    dealt to its CTAs and the free ones: their first boxes wait for the long solve to end, with a
    limit below that but above the time of its sweeps (0.5 ms holds about 60)."""
    cases = [inputs.flat_case(160, 96, 80, seed=9, tol=1e-9)] + \
            [inputs.flat_case(64, 48, 24 + i, seed=10 + i, tol=1e-9) for i in range(24)]
    solvers, alone = [], []
    for i, c in enumerate(cases):
        g = c.grid
        s = capi.Poisson(g.nx, g.ny, g.nz, g.h, inner_tol=1e-9 if i == 0 else 1e-4)
        s.set_density(c.F)
        assert "on chip" in s.describe(), s.describe()
        p = np.zeros(g.shape)
        assert s.solve(c.s, p, c.tol)[0] == capi.OK
        s.test_wait_limit(1e-3)
        solvers.append(s)
        alone.append(p)
    ps = [np.zeros(c.grid.shape) for c in cases]
    rcs = []
    for t in capi.batch_submit(solvers, [c.s for c in cases], ps, 1e-9):
        while True:
            rc, _ = capi.poll(t)
            if rc != capi.PENDING:
                break
        rcs.append(rc)
    for s in solvers:
        s.close()
    assert rcs == [capi.OK] * len(cases)
    for p, q in zip(ps, alone):
        assert np.linalg.norm(p - q) <= 2e-6 * np.linalg.norm(q)


@pytest.mark.parametrize("fine_pass", [1, 2, 3, 4])
def test_a_solve_after_a_fine_pass_timed_out_is_the_same_as_before(fine_pass):
    """512 tiles a pass, more blocks than are resident at once: the blocks of the first wave give up, those
    of the second find the solve ended and leave without a word to the reduction.  The next solve on
    the handle, of another source, gives bit for bit what it gave before."""
    c = inputs.flat_case(1024, 512, 8, seed=11, tol=1e-9)
    g = c.grid
    other = inputs.flat_case(1024, 512, 8, seed=12, tol=1e-9).s * 1e-3
    with capi.Poisson(g.nx, g.ny, g.nz, g.h, precond="mg") as s:
        s.set_density(c.F)
        ref = np.zeros(g.shape)
        rc, st_ref = s.solve(other, ref, c.tol)
        assert rc == capi.OK
        s.test_withhold_plane(fine_pass)
        p = np.zeros(g.shape)
        rc, _ = s.solve(c.s, p, c.tol, allow=(capi.ETIMEOUT,))
        assert rc == capi.ETIMEOUT and np.all(np.isfinite(p))
        assert s.test_counted_arrivals() == 0
        s.test_withhold_plane(0)
        p = np.zeros(g.shape)
        rc, st = s.solve(other, p, c.tol)
        assert rc == capi.OK
    assert st["outer_iters"] == st_ref["outer_iters"] and st["inner_iters"] == st_ref["inner_iters"]
    assert st["rel_residual"] == st_ref["rel_residual"] and np.array_equal(p, ref)


@pytest.mark.parametrize("fine_pass", [3, 4])
def test_applying_the_v_cycle_reports_a_timed_out_pass(fine_pass):
    """The V-cycle alone runs the restriction and the smoothing: a wait that runs out in one of them
    is told, and the next application gives what it gave before."""
    c = inputs.flat_case(64, 48, 32, seed=13)
    with capi.Poisson(64, 48, 32, c.grid.h, precond="mg") as s:
        s.set_density(c.F)
        r = np.random.default_rng(1).standard_normal(c.grid.shape)
        ref, z = np.empty_like(r), np.empty_like(r)
        s.precond_apply(r, ref, "mg", "fp32")
        s.test_withhold_plane(fine_pass)
        with pytest.raises(capi.PoissonError) as e:
            s.precond_apply(r, z, "mg", "fp32")
        assert e.value.status == capi.ETIMEOUT
        s.test_withhold_plane(0)
        s.precond_apply(r, z, "mg", "fp32")
        assert np.array_equal(z, ref)
