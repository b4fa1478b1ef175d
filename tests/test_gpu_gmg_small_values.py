"""Multigrid-preconditioned CG on a system of very small values: the V-cycle's FP32
vectors pass below 1.2e-38 before the solve is done, and have to keep what a
subnormal float holds.  Against the Jacobi solve in FP64 (whose numbers are all
normal), and in no more than twice the iterations of the same grid at ordinary
scale (an FP32 number of 1e-41 still has 12 bits, the V-cycle's needs are fewer)."""
import pytest

from paper_1704_02745_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_subnormal_vectors():
    from paper_1704_02745_gb300 import build, pb
    build.build()
    p = inputs.random_small(50, 33, 37, 29, n_atoms=30)

    def solve(ctx, scale, **kw):
        a = p.atoms.copy()
        a.q = a.q * scale
        with pb.Grid(ctx, p.grid, a) as g:
            phi = torch.zeros(p.grid.shape, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            info = g.solve(phi, check=False, precision="f64", max_iter=300, **kw)
            return info, phi

    with pb.Context(0) as ctx:
        ordinary, _ = solve(ctx, 1.0, precond="gmg", tol=1e-8)
        info, phi = solve(ctx, 1e-33, precond="gmg", tol=1e-8)
        _, want = solve(ctx, 1e-33, tol=1e-10)
    assert info.status == 0 and info.relres_true < 1e-8
    assert info.iterations <= 2 * ordinary.iterations
    assert float((phi - want).abs().max()) <= 1e-6 * float(want.abs().max())
