"""Grids of one context solved in turn, large and small ones by turns, and two
contexts in two threads: kernels whose shared memory follows the grid serve each
of them as when it is alone (the same bits)."""
import threading

import pytest

from paper_1704_02745_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(65, 65, 65), (9, 9, 9), (97, 61, 33), (20, 17, 40)]
MODES = [dict(precision="f64", precond="gmg"), dict(precision="f64"), dict(precision="f32_refine")]


@pytest.fixture(scope="module")
def pbm():
    from paper_1704_02745_gb300 import build, pb
    build.build()
    return pb


def solved(grid, shape, opts):
    phi = torch.zeros(shape, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    info = grid.solve(phi, tol=1e-9, **opts)
    assert info.status == 0 and info.iterations > 0
    return phi


def problems():
    return [inputs.random_small(80 + k, *s, n_atoms=12) for k, s in enumerate(SHAPES)]


@pytest.mark.parametrize("opts", MODES)
def test_in_turn(pbm, opts):
    probs = problems()
    with pbm.Context(0) as ctx:
        grids = [pbm.Grid(ctx, p.grid, p.atoms) for p in probs]
        first = [solved(g, p.grid.shape, opts) for g, p in zip(grids, probs)]
        for k in (0, 1, 2, 3, 1, 0, 3, 2):
            assert torch.equal(solved(grids[k], probs[k].grid.shape, opts), first[k]), SHAPES[k]
        for g in grids:
            g.close()


def test_in_threads(pbm):
    """Each thread plans and captures its launches again and again, beside the
    others' (every tensor is made beforehand: the threads call this library only)."""
    probs = problems()
    phis = [[[torch.zeros(p.grid.shape, dtype=torch.float64, device="cuda") for _ in range(5)] for _ in MODES]
            for p in probs]
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            with pbm.Context(0) as ctx:
                for m, opts in enumerate(MODES):
                    for phi in phis[k][m]:
                        with pbm.Grid(ctx, probs[k].grid, probs[k].atoms) as g:
                            g.solve(phi, tol=1e-9, **opts)
        except Exception as e:  # noqa: BLE001
            errors.append((SHAPES[k], repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(probs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for k in range(len(probs)):
        for m in range(len(MODES)):
            assert float(phis[k][m][0].abs().max()) > 0
            assert all(torch.equal(phi, phis[k][m][0]) for phi in phis[k][m]), (SHAPES[k], MODES[m])
