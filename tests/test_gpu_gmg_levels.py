"""Multigrid-preconditioned CG on the sizes where its levels change form: rows
with every remainder of four, no coarse level, one, a coarsest level too large
for the one-CTA kernel (a flat box), even sizes; packed, harmonic and explicit
operators, cold and warm.  Against the oracle's FP64 V-cycle: phi and E to 1e-8
at a true residual of 1e-10, iteration counts within its test's 15%, two at
least."""
import numpy as np
import pytest

import oracle
import oracle.gmg as G
from paper_1704_02745_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pbm():
    from paper_1704_02745_gb300 import build, pb
    build.build()
    pb.load()
    return pb


@pytest.mark.parametrize("opts", [{}, dict(eps_model="harmonic", coef="f32"), dict(coef="f64")])
@pytest.mark.parametrize("shape", [(3, 4, 5), (5, 7, 6), (8, 9, 10), (62, 61, 3), (19, 40, 34), (37, 18, 53)])
def test_levels(pbm, shape, opts):
    p = inputs.random_small(50 + shape[0], *shape, n_atoms=8 + shape[0])
    spec = p.grid.replace(**opts)
    s = oracle.setup(spec, p.atoms)
    ref = G.gmg_pcg(s, tol=1e-10)
    e_ref = oracle.energy(s, ref.phi)
    with pbm.Context(0) as ctx, pbm.Grid(ctx, spec, p.atoms) as g:
        phi = torch.zeros(spec.shape, dtype=torch.float64, device="cuda")
        info = g.solve(phi, precision="f64", precond="gmg", tol=1e-10)
        assert info.status == 0 and info.relres_true < 2e-10
        assert float(np.max(np.abs(phi.cpu().numpy() - ref.phi))) <= 1e-8 * np.max(np.abs(ref.phi))
        assert abs(g.energy(phi) - e_ref) <= 1e-8 * abs(e_ref)
        assert abs(info.iterations - ref.iters) <= max(2, 0.15 * ref.iters)
        # from a point near the solution
        start = phi.clone()
        phi.mul_(1.0 + 1e-3)
        info = g.solve(phi, precision="f64", precond="gmg", tol=1e-10, warm_start=True)
        assert info.status == 0 and info.iterations <= ref.iters
        assert float((phi - start).abs().max()) <= 1e-8 * float(start.abs().max())
