"""The resident form of a solve (whole inner solves in one cooperative kernel)
against the tick form (poll_every > 0 asks for it) and the oracle: row lengths
with every remainder of four, one to many bricks per axis, every coefficient
storage, both precisions, with and without wrap, plain CG, the iteration cap,
and solves running at the same time.

Tolerances: both forms stop at a true residual of 1e-10 relative; the oracle
comparison is the one of the FP64 parity tests (1e-8 of max|phi| and of |E|),
which leaves two digits for the condition of these grids; a refined solve's
last inner residual may differ by the summation order, so its two forms are
held to the same bound.  Iteration counts of FP64 solves: the FP64 tests' 2%, two
at least (FP32 inner solves have none to hold to: their counts follow the
rounding of each form)."""
import threading

import numpy as np
import pytest

import oracle
from paper_1704_02745_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pbm():
    from paper_1704_02745_gb300 import build, pb
    build.build()
    pb.load()
    return pb


@pytest.fixture(scope="module")
def ctx(pbm):
    c = pbm.Context(0)
    yield c
    c.close()


def zeros(shape):
    return torch.zeros(shape, dtype=torch.float64, device="cuda")


def rel_max(a, b):
    return float((a - b).abs().max() / b.abs().max())


# (nx, ny, nz): one brick, partial groups of four, few and many planes a
# brick, more rows than a brick holds, a grid the register builds cannot hold
SHAPES = [(5, 3, 3), (8, 7, 1), (17, 5, 40), (30, 61, 9), (47, 45, 50), (64, 21, 97), (131, 37, 29), (97, 81, 113)]


@pytest.mark.parametrize("precision", ["f64", "f32_refine"])
@pytest.mark.parametrize("shape", SHAPES)
def test_matches_tick_form_and_oracle(pbm, ctx, shape, precision):
    p = inputs.random_small(31 + shape[0], *shape, n_atoms=10 + shape[0])
    if min(shape) == 1:  # a planar grid: every atom on its plane of nodes, h apart at most
        p.atoms.xyz[:, int(np.argmin(shape))] = 0.0
        with pytest.raises(pbm.PbError):  # a trilinear cell needs two planes: refused as before
            pbm.Grid(ctx, p.grid, p.atoms)
        return
    s = oracle.setup(p.grid, p.atoms)
    ref = oracle.pcg(s, tol=1e-12)
    e_ref = oracle.energy(s, ref.phi)
    with pbm.Grid(ctx, p.grid, p.atoms) as g:
        out = []
        for poll in (0, 8):
            phi = zeros(p.grid.shape)
            info = g.solve(phi, precision=precision, tol=1e-10, poll_every=poll)
            assert info.status == 0 and info.relres_true < 1e-10
            assert abs(g.energy(phi) - e_ref) <= 1e-8 * abs(e_ref)
            assert float(np.max(np.abs(phi.cpu().numpy() - ref.phi))) <= 1e-8 * np.max(np.abs(ref.phi))
            out.append((phi, info))
        assert rel_max(out[0][0], out[1][0]) <= 1e-8
        if precision == "f64":
            assert abs(out[0][1].iterations - out[1][1].iterations) <= max(2, 0.02 * out[1][1].iterations)
        # again: bit for bit
        phi = zeros(p.grid.shape)
        info = g.solve(phi, precision=precision, tol=1e-10)
        assert info.iterations == out[0][1].iterations and torch.equal(phi, out[0][0])


OPTIONS = [dict(coef="f32"), dict(coef="bf16"), dict(coef="f64"), dict(coef="f32", eps_model="harmonic"),
           dict(coef="bf16", eps_model="harmonic"), dict(periodic=True, kappa_mask=False),
           dict(periodic=True, kappa_mask=False, coef="f32"), dict(periodic=True, kappa_mask=False, coef="bf16")]
# (lambda = 1 on the periodic grids: the atoms cover every node of the smallest,
# and without a node in the solvent a periodic A is singular)


@pytest.mark.parametrize("opts", OPTIONS)
@pytest.mark.parametrize("shape", [(4, 5, 3), (35, 22, 19), (66, 41, 58)])
def test_storages_and_wrap(pbm, ctx, shape, opts):
    p = inputs.random_small(7 + shape[0], *shape, n_atoms=6 + shape[0])
    spec = p.grid.replace(**opts)
    with pbm.Grid(ctx, spec, p.atoms) as g:
        for precision in ("f32_refine", "f64"):
            for precond in ("jacobi", "none"):
                out = []
                for poll in (0, 8):
                    phi = zeros(spec.shape)
                    info = g.solve(phi, precision=precision, precond=precond, tol=1e-10, poll_every=poll)
                    assert info.status == 0 and info.relres_true < 1e-10
                    out.append((phi, info))
                assert rel_max(out[0][0], out[1][0]) <= 1e-8, (precision, precond)
                if precision == "f64":
                    assert abs(out[0][1].iterations - out[1][1].iterations) <= max(2, 0.02 * out[1][1].iterations)


@pytest.mark.parametrize("precision", ["f64", "f32", "f32_refine"])
@pytest.mark.parametrize("cap", [0, 1, 7])
def test_iteration_cap(pbm, ctx, precision, cap):
    p = inputs.random_small(12, 40, 33, 27, n_atoms=60)
    with pbm.Grid(ctx, p.grid, p.atoms) as g:
        infos = [g.solve(zeros(p.grid.shape), check=False, precision=precision, tol=1e-12, max_iter=cap,
                         poll_every=poll) for poll in (0, 8)]
    assert infos[0].status == infos[1].status == pbm.PB_ERR_NOT_CONVERGED
    assert infos[0].iterations == infos[1].iterations
    assert abs(infos[0].relres - infos[1].relres) <= 1e-5 * infos[1].relres


def test_solves_at_the_same_time(pbm, ctx):
    """Two contexts in two threads and a server: cooperative launches of several
    streams beside a server's graphs; every result as when alone."""
    p = inputs.random_small(40, 90, 70, 60, n_atoms=150)
    snaps = inputs.snapshot_batch(count=8)

    def alone(c):
        with pbm.Grid(c, p.grid, p.atoms) as g:
            phi = zeros(p.grid.shape)
            g.solve(phi, precision="f32_refine", tol=1e-9)
            return phi

    want = alone(ctx)
    errors = []

    def work():
        try:
            with pbm.Context(0) as c:
                for _ in range(6):
                    if not torch.equal(alone(c), want):
                        errors.append("another result")
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    with pbm.Server(ctx, 8 << 30, tol=1e-9, inner_tol=1e-4, warm_start=False) as srv:
        first = [srv.poll(t, 60000)[0].energy for t in
                 [srv.submit(k, s.grid, s.atoms) for k, s in enumerate(snaps)]]
        threads = [threading.Thread(target=work) for _ in range(2)]
        for t in threads:
            t.start()
        for _ in range(3):
            tickets = [srv.submit(k, s.grid, s.atoms) for k, s in enumerate(snaps)]
            again = [srv.poll(t, 60000)[0].energy for t in tickets]
            assert again == first
        for t in threads:
            t.join()
    assert not errors
