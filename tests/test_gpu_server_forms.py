"""A served solve runs on the chip or in phase ticks by its grid's size alone, so
its result is the same bits alone and beside any others: small grids beside one
too large for the chip and beside ones whose rows are too long for it, with and
without wrap; and a server made for ticks (poll_every > 0), whose form serves
every large grid and mixed batch, alone and in a mix, against the oracle.

Energies against the oracle: relative 1e-7 at a true residual of 1e-9, the
fault tests' bound."""
import pytest

import oracle
from paper_1704_02745_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

OPTS = dict(tol=1e-9, inner_tol=1e-4, warm_start=False)


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
    p = inputs.random_small(170 + k, *shape, n_atoms=10 + 3 * k)
    return p.grid.replace(**kw), p.atoms


def key(r):
    return r.status, r.energy, r.info.iterations, r.info.relres, r.info.relres_true


def alone_and_mixed(srv, probs, rounds=3):
    """Results one at a time; then all together, `rounds` times over, a submission at a time."""
    alone = [srv.poll(srv.submit(k, *p), 60000)[0] for k, p in enumerate(probs)]
    for r in range(rounds):
        order = [(k + r) % len(probs) for k in range(len(probs))]
        tickets = [(k, srv.submit(1000 * r + k, *probs[k])) for k in order]
        for k, t in tickets:
            assert key(srv.poll(t, 120000)[0]) == key(alone[k]), probs[k][0].shape
    return alone


@pytest.mark.parametrize("periodic", [False, True])
def test_small_beside_large(pbm, ctx, periodic):
    kw = dict(periodic=True, kappa_mask=False) if periodic else {}
    shapes = [(33, 40, 50), (61, 16, 97), (20, 23, 31), (97, 49, 65), (257, 193, 181), (2060, 5, 7), (2100, 9, 4)]
    probs = [problem(k, s, **kw) for k, s in enumerate(shapes)]
    with pbm.Server(ctx, 16 << 30, **OPTS) as srv:
        alone = alone_and_mixed(srv, probs)
    assert all(r.status == 0 and r.info.relres_true < 1.01e-9 for r in alone)


@pytest.mark.parametrize("periodic", [False, True])
def test_ticks_alone_and_in_a_mix(pbm, ctx, periodic):
    kw = dict(periodic=True, kappa_mask=False) if periodic else {}
    shapes = [(17, 20, 33), (33, 33, 33), (60, 21, 40), (5, 44, 9), (66, 18, 25)]
    probs = [problem(k, s, **kw) for k, s in enumerate(shapes)]
    probs += [problem(k + 10, (25, 26, 27), **kw) for k in range(20)]
    with pbm.Server(ctx, 8 << 30, poll_every=8, **OPTS) as srv:
        alone = alone_and_mixed(srv, probs, rounds=2)
    with pbm.Server(ctx, 8 << 30, **OPTS) as srv:
        chip = [srv.poll(srv.submit(k, *p), 60000)[0] for k, p in enumerate(probs)]
    assert any(key(a) != key(b) for a, b in zip(alone, chip))  # (two forms: other groupings of the sums)
    for k, (grid, atoms) in enumerate(probs[:8]):
        s = oracle.setup(grid, atoms)
        want = oracle.energy(s, oracle.pcg(s, tol=1e-11).phi)
        assert alone[k].status == 0 and abs(alone[k].energy - want) <= 1e-7 * abs(want)


def test_measuring_a_server_of_small_grids(pbm, ctx):
    """Between profile_begin and profile_end solves run in the ticks that are timed;
    before and after in their own form."""
    probs = [problem(k, (33, 40, 20 + k)) for k in range(6)]
    with pbm.Server(ctx, 8 << 30, **OPTS) as srv:
        first = [srv.poll(srv.submit(k, *p), 60000)[0] for k, p in enumerate(probs)]
        srv.profile_begin()
        timed = [srv.poll(t, 60000)[0] for t in [srv.submit(k, *p) for k, p in enumerate(probs)]]
        prof = srv.profile_end()
        again = [srv.poll(t, 60000)[0] for t in [srv.submit(k, *p) for k, p in enumerate(probs)]]
    assert prof.launches_stencil > 0 and prof.launches_update > 0 and prof.launches_resid > 0
    for a, b, c in zip(first, timed, again):
        assert key(a) == key(c) and b.status == 0 and abs(b.energy - a.energy) <= 2e-7 * abs(a.energy)
