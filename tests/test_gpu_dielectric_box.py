"""The dielectric map's boxes and FP32 test against the oracle, bit for bit: spheres
whose surface meets nodes and midpoints exactly, within rounding of them and within
the FP32 test's margin; spheres smaller than a spacing and larger than the grid;
atoms far from the coordinate origin; with and without wrap."""
import numpy as np
import pytest

import oracle
from paper_1704_02745_gb300 import inputs

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def lattice():
    p = inputs.random_small(61, 22, 27, 19, n_atoms=120)
    rng = np.random.default_rng(61)
    half = rng.integers(6, 2 * np.array([22, 27, 19]) - 7, size=(120, 3)) / 2
    p.atoms.xyz = np.asarray(p.grid.origin) + p.grid.h * half
    p.atoms.r = p.grid.h * rng.choice([0.5, 1.0, np.sqrt(0.5), 1.5, np.sqrt(2.0), 2.0], 120)
    p.atoms.r += rng.choice([0.0, 1e-15, -1e-15, 1e-6, -1e-6, 1e-4, -1e-4], 120)
    return p


def sizes():
    p = inputs.random_small(62, 33, 14, 25, n_atoms=5)
    p.atoms.r = np.array([0.01, 9.0, 0.2, 30.0, 1.0])
    return p


def far():
    p = inputs.random_small(63, 21, 18, 26, n_atoms=90)
    p.atoms.xyz = p.atoms.xyz + 3e4
    p.grid = p.grid.replace(origin=tuple(o + 3e4 for o in p.grid.origin))
    return p


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("maker", [lattice, sizes, far])
def test_map_bit_exact(maker, periodic):
    from paper_1704_02745_gb300 import build, pb
    build.build()
    p = maker()
    if periodic and maker is sizes:  # (an image of a sphere must not meet itself)
        p.atoms.r = np.minimum(p.atoms.r, 3.0)
    spec = p.grid.replace(periodic=periodic)
    s = oracle.setup(spec, p.atoms)
    with pb.Context(0) as ctx, pb.Grid(ctx, spec, p.atoms) as g:
        assert np.array_equal(g.export("eps_x"), s.ex)
        assert np.array_equal(g.export("eps_y"), s.ey)
        assert np.array_equal(g.export("eps_z"), s.ez)
        assert np.array_equal(g.export("lambda"), s.lam)
