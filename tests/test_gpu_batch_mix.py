"""Batches whose jobs take different kernels: solves that join a running batch of streamed grids, and
batches that gain their first streamed or their first on-chip job while they run; and two threads that
solve on streams of their own, whose persistent launches must not meet on the GPU."""
import threading

import numpy as np
import pytest

import oracle
from paper_1410_1942_gb300 import build, capi, inputs

pytestmark = pytest.mark.gpu

L2_TOL = 1e-6
TILE = 12012204  # a streamed one-sweep tile: small grids with it take no on-chip launch


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available()
    build.build()
    capi.load()


def _solver(c, tile):
    g = c.grid
    s = capi.Poisson(g.nx, g.ny, g.nz, g.h, tile=tile)
    s.set_density(c.F)
    assert ("on chip" in s.describe()) == (tile == 0), s.describe()
    return s


def _poll_all(tickets):
    done = {}
    while len(done) < len(tickets):
        for t in tickets:
            if t not in done:
                rc, _ = capi.poll(t)
                if rc != capi.PENDING:
                    done[t] = rc
    return [done[t] for t in tickets]


def _join(cases, tiles, first):
    """Submits the first jobs, runs one refinement step of them, then submits the others."""
    solvers = [_solver(c, t) for c, t in zip(cases, tiles)]
    ps = [np.zeros(c.grid.shape) for c in cases]
    a = capi.batch_submit(solvers[:first], [c.s for c in cases[:first]], ps[:first], 1e-9)
    assert capi.poll(a[0])[0] == capi.PENDING
    b = capi.batch_submit(solvers[first:], [c.s for c in cases[first:]], ps[first:], 1e-9)
    rcs = _poll_all(a + b)
    for s in solvers:
        s.close()
    assert rcs == [capi.OK] * len(cases)
    for c, p in zip(cases, ps):
        op, rhs = oracle.operator(c.F), oracle.rhs(c.s, c.grid.h)
        assert oracle.rel_residual(op, rhs, p) <= 1e-9 * (1 + 1e-6)
        ref = oracle.pcg(op, rhs, tol=1e-12, precond="ssor").x
        assert np.linalg.norm(p - ref) <= L2_TOL * np.linalg.norm(ref)


def _cases(shapes):
    return [inputs.flat_case(*s, seed=40 + i, tol=1e-9) for i, s in enumerate(shapes)]


EVEN = [(64, 48, 32), (32, 32, 32), (72, 40, 24)]
ODD = [(61, 47, 30), (37, 23, 19), (50, 33, 26)]  # rows at a pitch


@pytest.mark.parametrize("tile", [TILE, 12204])
def test_solves_join_a_running_batch_of_streamed_grids(tile):
    _join(_cases(EVEN + EVEN), [tile] * 6, 3)


def test_odd_rows_join_a_running_batch_of_streamed_grids():
    """The joint launch changes to the kernel for rows of any length while it holds plain rows."""
    _join(_cases(EVEN + ODD), [TILE] * 6, 3)


@pytest.mark.parametrize("tiles", [[0] * 3 + [TILE] * 3, [TILE] * 3 + [0] * 3,
                                   [0, TILE, 0, TILE, 0, TILE]])
def test_streamed_and_on_chip_jobs_join_each_other(tiles):
    _join(_cases(EVEN + ODD), tiles, 3)


def test_a_streamed_solve_alone_and_in_the_mix_agree():
    cases = _cases(EVEN + ODD)
    alone = np.zeros(cases[2].grid.shape)
    with _solver(cases[2], TILE) as s:
        assert s.solve(cases[2].s, alone, 1e-9)[0] == capi.OK
    solvers = [_solver(c, TILE) for c in cases]
    ps = [np.zeros(c.grid.shape) for c in cases]
    rcs = _poll_all(capi.batch_submit(solvers, [c.s for c in cases], ps, 1e-9))
    for s in solvers:
        s.close()
    assert rcs == [capi.OK] * len(cases)
    assert np.linalg.norm(ps[2] - alone) <= 2 * L2_TOL * np.linalg.norm(alone)


@pytest.mark.parametrize("tiles", [(0, 0), (TILE, TILE), (0, TILE)])
def test_two_threads_solve_on_their_own_streams(tiles):
    """Both solves launch kernels that need all their CTAs resident; ordered one after another, each
    gives what it gives alone, bit for bit."""
    import torch
    cases = _cases([(128, 64, 48), (96, 64, 64)])
    streams = [torch.cuda.Stream() for _ in cases]
    solvers, alone = [], []
    for c, tile, st in zip(cases, tiles, streams):
        g = c.grid
        s = capi.Poisson(g.nx, g.ny, g.nz, g.h, tile=tile, stream=st)
        s.set_density(c.F)
        p = np.zeros(g.shape)
        assert s.solve(c.s, p, 1e-9)[0] == capi.OK
        solvers.append(s)
        alone.append(p)
    same = [0, 0]

    def work(q):
        for _ in range(5):
            p = np.zeros(cases[q].grid.shape)
            rc, _ = solvers[q].solve(cases[q].s, p, 1e-9, allow=(capi.OK, capi.ETIMEOUT))
            same[q] += rc == capi.OK and np.array_equal(p, alone[q])

    threads = [threading.Thread(target=work, args=(q,)) for q in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s in solvers:
        s.close()
    assert same == [5, 5]
