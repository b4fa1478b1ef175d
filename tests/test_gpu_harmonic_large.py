"""The harmonic-average edges of spheres of tens of angstrom on grids of some
hundred, bit for bit against the oracle: each grid is a slab with one sphere that
leaves a few thousandths of one edge uncovered, where an FP32 test of the squared
distance is off by several thousandths of a square angstrom."""
import numpy as np
import pytest

import oracle
from paper_1704_02745_gb300 import inputs

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def slab(seed, n, h, radius):
    """One sphere whose surface cuts off less than 4e-3 A at each end of a y-edge."""
    rng = np.random.default_rng(seed)
    ny, nz = 5, 33
    while True:
        i, j, k = int(rng.integers(n // 2, n - 1)), int(rng.integers(0, ny - 1)), int(rng.integers(0, nz))
        half = h / 2 - rng.uniform(2e-4, 4e-3)  # of the chord along the edge
        ang = rng.uniform(-0.3, 0.3) + (0 if rng.random() < 0.5 else np.pi)
        d = np.sqrt(radius * radius - half * half)
        centre = np.array([i * h + d * np.cos(ang), (j + 0.5) * h, k * h + d * np.sin(ang)])
        if 0 < centre[0] < (n - 1) * h and 0 < centre[2] < (nz - 1) * h:  # an atom lies in the grid
            break
    p = inputs.random_small(1, n, ny, nz, h=h, n_atoms=1)
    p.grid = p.grid.replace(origin=(0.0, 0.0, 0.0), eps_model="harmonic", coef="f64")
    p.atoms.xyz, p.atoms.r = centre[None, :], np.array([radius])
    return p, (i, j, k)


CASES = [((230, 404, 519, 568, 606, 785, 945, 948, 1012, 1284, 1360, 1460), 513, 1.07, 60.0), (tuple(range(12)), 401, 0.613, 60.0), (tuple(range(12)), 257, 0.61, 30.0)]


@pytest.mark.parametrize("seeds,n,h,radius", CASES)
def test_edges_bit_exact(seeds, n, h, radius):
    from paper_1704_02745_gb300 import build, pb
    build.build()
    with pb.Context(0) as ctx:
        for seed in seeds:
            p, _ = slab(seed, n, h, radius)
            s = oracle.setup(p.grid, p.atoms)
            with pb.Grid(ctx, p.grid, p.atoms) as g:
                for name, want in (("eps_x", s.ex), ("eps_y", s.ey), ("eps_z", s.ez)):
                    assert np.array_equal(g.export(name), want), (seed, name)
