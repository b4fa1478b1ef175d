"""The dielectric map of spheres far smaller than the grid's spacing, bit for bit
against the oracle: every sphere's surface passes within a few 1e-4 A of a node or
of an edge's midpoint, where offsets of FP32 from a box's first node are off by
as much."""
import numpy as np
import pytest

import oracle
from paper_1704_02745_gb300 import inputs

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def coarse(h, seed):
    p = inputs.random_small(64, 20, 18, 23, h=h, n_atoms=400)
    rng = np.random.default_rng(seed)
    half = rng.integers(4, 2 * np.array([20, 18, 23]) - 6, size=(400, 3))
    half[np.arange(400), rng.integers(0, 3, 400)] //= 2  # at most one odd coordinate is a midpoint
    odd = half % 2
    odd[:, 1] &= 1 - odd[:, 0]
    odd[:, 2] &= 1 - (odd[:, 0] | odd[:, 1])
    half = half // 2 * 2 + odd
    u = rng.normal(size=(400, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    p.atoms.r = rng.uniform(0.8, 2.0, 400)
    dist = p.atoms.r + rng.uniform(-4e-4, 4e-4, 400)
    p.atoms.xyz = np.asarray(p.grid.origin) + h / 2 * half + u * dist[:, None]
    return p


@pytest.mark.parametrize("h", [300.0, 3000.0, 30000.0])
def test_map_bit_exact(h):
    from paper_1704_02745_gb300 import build, pb
    build.build()
    with pb.Context(0) as ctx:
        for seed in range(4):
            p = coarse(h, seed)
            s = oracle.setup(p.grid, p.atoms)
            assert 100 < np.count_nonzero(s.ex != 80.0) + np.count_nonzero(s.ey != 80.0) + np.count_nonzero(s.ez != 80.0)
            with pb.Grid(ctx, p.grid, p.atoms) as g:
                for name, want in (("eps_x", s.ex), ("eps_y", s.ey), ("eps_z", s.ez), ("lambda", s.lam)):
                    assert np.array_equal(g.export(name), want), (h, seed, name)
