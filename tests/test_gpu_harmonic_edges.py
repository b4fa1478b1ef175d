"""The harmonic-average edge kernel against the oracle, bit for bit, where its
search can go wrong: more atoms at an edge than it collects at once, spheres that
end exactly on nodes or within the FP32 test's margin of them, atoms far from the
coordinate origin, cells of a few large spheres, no atom near most edges."""
import numpy as np
import pytest

import oracle
from paper_1704_02745_gb300 import inputs

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def crowded():
    return inputs.random_small(31, 17, 15, 19, n_atoms=2500)


def on_nodes():
    p = inputs.random_small(32, 18, 21, 16, n_atoms=60)
    rng = np.random.default_rng(32)
    n = np.array([18, 21, 16])
    node = rng.integers(2, n - 2, size=(60, 3))
    p.atoms.xyz = np.asarray(p.grid.origin) + p.grid.h * node
    p.atoms.r = p.grid.h * rng.choice([1.0, 1.5, 2.0, 3.0], 60) + rng.choice([0.0, 5e-4, -5e-4, 2e-3, -2e-3], 60)
    return p


def far():
    p = inputs.random_small(33, 20, 17, 23, n_atoms=150)
    p.atoms.xyz = p.atoms.xyz + 3e4
    p.grid = p.grid.replace(origin=tuple(o + 3e4 for o in p.grid.origin))
    return p


def large_spheres():
    p = inputs.random_small(34, 40, 9, 33, n_atoms=6)
    p.atoms.r = np.array([0.3, 6.0, 0.7, 1.0, 0.2, 2.5])
    return p


def one_atom():
    return inputs.random_small(35, 65, 30, 41, n_atoms=1)


@pytest.mark.parametrize("maker", [crowded, on_nodes, far, large_spheres, one_atom])
def test_edges_bit_exact(maker):
    from paper_1704_02745_gb300 import build, pb
    build.build()
    p = maker()
    spec = p.grid.replace(eps_model="harmonic", coef="f64")
    s = oracle.setup(spec, p.atoms)
    with pb.Context(0) as ctx, pb.Grid(ctx, spec, p.atoms) as g:
        assert np.array_equal(g.export("eps_x"), s.ex)
        assert np.array_equal(g.export("eps_y"), s.ey)
        assert np.array_equal(g.export("eps_z"), s.ez)
