"""A server's round holds 192 iterations of a grid at most, however many its solve
takes: a solve of many iterations takes three launches (residual pass, inner
solves, residual pass) for each 192 of them, and goes on from round to round
where it stopped.  Plain FP32 solves are one inner solve; a refined solve of the
same system ends at the true residual it asks for, and its energy is held to a
plain FP64 solve's at 1e-7, the fault tests' bound.  (Plain FP32 has no such bound:
its recursive residual says nothing of the error on a system this ill-conditioned.)"""
import numpy as np
import pytest

from paper_1704_02745_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,kw", [((97, 81, 60), {}), ((33, 30, 29), {}), ((5, 4, 600), {}),
                                      ((60, 41, 50), dict(periodic=True, kappa_mask=False))])
@pytest.mark.parametrize("precision", ["f32", "f32_refine"])
def test_long_solves(shape, kw, precision):
    from paper_1704_02745_gb300 import build, pb
    build.build()
    p = inputs.random_small(9, *shape, n_atoms=40, ionic_strength=1e-3, eps_out=300.0)
    p.atoms.q = np.abs(p.atoms.q) + 0.2
    spec = p.grid.replace(**kw)
    tol = 1e-6 if precision == "f32" else 1e-9
    opts = dict(precision=precision, precond="none", tol=tol, inner_tol=1e-9, warm_start=False)
    with pb.Context(0) as ctx:
        with pb.Grid(ctx, spec, p.atoms) as g:
            phi = torch.zeros(spec.shape, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            g.solve(phi, precision="f64", tol=1e-11)
            want = g.energy(phi)
        with pb.Server(ctx, 8 << 30, **opts) as srv:
            before = ctx.stats()[0]
            alone = srv.poll(srv.submit(0, spec, p.atoms), 60000)[0]
            launches = ctx.stats()[0] - before
            assert alone.status == 0
            if precision == "f32_refine":
                assert alone.info.relres_true < 1.01 * tol and abs(alone.energy - want) <= 1e-7 * abs(want)
            assert alone.info.iterations > 200
            # (a refined solve's inner solves each end in a round of their own)
            assert launches >= 3 * (alone.info.iterations // 192)
            many = [srv.poll(t, 60000)[0] for t in [srv.submit(k, spec, p.atoms) for k in range(1, 9)]]
    for r in many:
        assert (r.energy, r.info.iterations, r.info.relres) == (alone.energy, alone.info.iterations, alone.info.relres)
