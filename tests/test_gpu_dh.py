"""The FP64 Debye-Hueckel boundary sum against the oracle, node by node: no salt,
ordinary salt, screening so strong that the far terms underflow, atoms far from
the coordinate origin, and atom counts around the kernel's tiles; faces of
short and long lines.

All charges are positive, so a node's error is bounded by its terms': a term
carries a few roundings and its exponent kappa r one more, in the oracle and
here, and n terms add n roundings: (n + 8 + 2 kappa r) 2^-53 each side.  Values
below 1e-290 (underflowed terms) are compared absolutely."""
import math

import numpy as np
import pytest

import oracle
from paper_1704_02745_gb300 import inputs

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_atoms", [1, 255, 257])
@pytest.mark.parametrize("ionic,shift", [(0.0, 0.0), (0.15, 0.0), (2.0, 3e4), (1e5, 0.0)])
def test_ghost_values(n_atoms, ionic, shift):
    from paper_1704_02745_gb300 import build, pb
    build.build()
    p = inputs.random_small(90 + n_atoms, 19, 13, 9, n_atoms=n_atoms, ionic_strength=ionic)
    p.atoms.q = np.abs(p.atoms.q) + 0.01
    p.atoms.xyz = p.atoms.xyz + shift
    spec = p.grid.replace(origin=tuple(o + shift for o in p.grid.origin))
    want = oracle.setup(spec, p.atoms).ghost
    with pb.Context(0) as ctx, pb.Grid(ctx, spec, p.atoms) as g:
        got = g.export("ghost")
    r_max = spec.h * math.sqrt(20 ** 2 + 14 ** 2 + 10 ** 2)
    kappa = math.sqrt(ionic) / 3.04  # Debye length 3.04 A / sqrt(I) in water
    tol = 2 * (n_atoms + 8 + 2 * 1.2 * kappa * r_max) * 2.0 ** -53
    if shift:  # r from coordinates rounded at 3e4: the same differences in both, exact subtractions
        tol *= 2
    assert np.all(np.abs(got - want) <= tol * np.abs(want) + 1e-290)


@pytest.mark.parametrize("shape", [(6, 7, 40), (33, 5, 6), (16, 31, 32), (65, 15, 17), (3, 70, 5)])
@pytest.mark.parametrize("n_atoms", [63, 64, 130])
def test_line_lengths(n_atoms, shape):
    from paper_1704_02745_gb300 import build, pb
    build.build()
    p = inputs.random_small(sum(shape), *shape, n_atoms=n_atoms, ionic_strength=0.15)
    p.atoms.q = np.abs(p.atoms.q)
    p.atoms.q[0] = 0.0
    want = oracle.setup(p.grid, p.atoms).ghost
    with pb.Context(0) as ctx, pb.Grid(ctx, p.grid, p.atoms) as g:
        got = g.export("ghost")
    r_max = p.grid.h * math.sqrt(sum((n + 1) ** 2 for n in shape))
    tol = 2 * (n_atoms + 8 + 2 * 1.2 * math.sqrt(0.15) / 3.04 * r_max) * 2.0 ** -53
    assert np.all(np.abs(got - want) <= tol * np.abs(want))
