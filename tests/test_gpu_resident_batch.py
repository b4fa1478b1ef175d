"""Whole inner solves of a server's grids, side by side in cooperative launches:
grids at the edges of the plans (one group of x nodes, one plane, the widest and
deepest bricks, one brick and many), with and without wrap, and batches that
change between this form and phase ticks.

Energies E = 1/2 phi.b of a solution with residual r are off by 1/2 phi.r, at most
|phi| |r| / (phi.b) relative; with all charges positive phi at the charges is at
least its rms value, so that |phi| |b| / (phi.b) <= sqrt(N / atoms) times the
spread of the charges (1.2 here), and the bound is 3 tol sqrt(N / atoms).  A
grid's plan and the order of its sums do not depend on what else runs, so its
result is the same bits alone and in any batch."""
import math

import numpy as np
import pytest

from paper_1704_02745_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-9
SHAPES = [(3, 4, 5), (4, 3, 29), (5, 33, 9), (29, 8, 8), (33, 33, 33), (61, 16, 97), (97, 81, 113), (257, 20, 30),
          (129, 97, 65)]


@pytest.fixture(scope="module")
def pbm():
    from paper_1704_02745_gb300 import build, pb
    build.build()
    return pb


@pytest.fixture(scope="module")
def ctx(pbm):
    with pbm.Context(0) as c:
        yield c


def problem(k, shape, **kw):
    p = inputs.random_small(70 + k, *shape, n_atoms=5 + 3 * k)
    p.atoms.q = np.abs(p.atoms.q) + 0.3
    return p.grid.replace(**kw), p.atoms


def bound(grid, atoms):
    return 3 * TOL * math.sqrt(np.prod(grid.shape) / len(atoms.q))


def reference(pbm, ctx, grid, atoms):
    with pbm.Grid(ctx, grid, atoms) as g:
        phi = torch.zeros(grid.shape, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        g.solve(phi, precision="f64", tol=1e-11)
        return g.energy(phi)


def same(a, b):
    return (a.energy, a.info.iterations, a.info.relres) == (b.energy, b.info.iterations, b.info.relres)


@pytest.mark.parametrize("periodic", [False, True])
def test_alone_and_together(pbm, ctx, periodic):
    kw = dict(periodic=periodic)
    if periodic:
        kw["kappa_mask"] = False  # (no node of the smallest grids lies outside the atoms: A would be singular)
    probs = [problem(k, s, **kw) for k, s in enumerate(SHAPES)]
    with pbm.Server(ctx, 8 << 30, tol=TOL, inner_tol=1e-4, warm_start=False) as srv:
        alone = [srv.poll(srv.submit(k, *p), 60000)[0] for k, p in enumerate(probs)]
        tickets = [srv.submit(k, *p) for k, p in enumerate(probs)] + [srv.submit(100 + k, *p) for k, p in enumerate(probs)]
        together = [srv.poll(t, 60000)[0] for t in tickets]
    for k, p in enumerate(probs):
        want = reference(pbm, ctx, *p)
        assert alone[k].status == 0 and alone[k].info.relres_true < 1.01 * TOL, SHAPES[k]
        assert abs(alone[k].energy - want) <= bound(*p) * abs(want), SHAPES[k]
        assert same(together[k], alone[k]) and same(together[len(probs) + k], alone[k]), SHAPES[k]


def test_beside_a_grid_that_needs_ticks(pbm, ctx):
    """A grid too large to stay on the chip turns the batch to ticks, from
    whatever state the others are in; later solves run whole again."""
    small = [problem(k, (33 + 8 * k, 40, 50)) for k in range(6)]
    large = problem(9, (257, 193, 181))
    with pbm.Server(ctx, 16 << 30, tol=TOL, inner_tol=1e-4, warm_start=False) as srv:
        alone = [srv.poll(srv.submit(k, *p), 60000)[0] for k, p in enumerate(small)]
        tickets = []
        for k, p in enumerate(small):
            tickets.append(srv.submit(k, *p))
            if k == 2:
                big = srv.submit(50, *large)
        mixed = [srv.poll(t, 60000)[0] for t in tickets]
        res = srv.poll(big, 60000)[0]
        again = [srv.poll(srv.submit(k, *p), 60000)[0] for k, p in enumerate(small)]
    assert res.status == 0 and res.info.relres_true < 1.01 * TOL
    want = reference(pbm, ctx, *large)
    assert abs(res.energy - want) <= bound(*large) * abs(want)
    for k in range(len(small)):
        assert mixed[k].status == 0 and abs(mixed[k].energy - alone[k].energy) <= 2 * bound(*small[k]) * abs(alone[k].energy)
        assert same(again[k], alone[k])


def test_more_grids_than_a_launch_holds(pbm, ctx):
    grid, atoms = problem(3, (29, 23, 31))
    with pbm.Server(ctx, 8 << 30, tol=TOL, inner_tol=1e-4, warm_start=False) as srv:
        alone = srv.poll(srv.submit(0, grid, atoms), 60000)[0]
        res = [srv.poll(t, 60000)[0] for t in [srv.submit(k, grid, atoms) for k in range(70)]]
    assert all(same(r, alone) for r in res)
