"""The FP64 Debye-Hueckel sum on a grid so long that one charge's terms run from
ordinary values through every range of the kernel's quotient down to underflow
(kappa r up to 760): node by node against the oracle.  A term carries a few
roundings and its exponent one more: (9 + 2 kappa r) 2^-53 a side, and what lies
below 1e-290 is compared absolutely."""
import math

import numpy as np
import pytest

import oracle
from paper_1704_02745_gb300 import inputs

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 2])
def test_one_charge_on_a_long_grid(axis):
    from paper_1704_02745_gb300 import build, pb
    build.build()
    shape = [4, 3, 3]
    shape[axis] = 6000
    p = inputs.random_small(5, *shape, h=1.0, n_atoms=1, ionic_strength=0.15)
    p.grid = p.grid.replace(origin=(0.0, 0.0, 0.0))
    p.atoms.xyz = np.full((1, 3), 1.3)
    p.atoms.q = np.array([0.7])
    want = oracle.setup(p.grid, p.atoms).ghost
    with pb.Context(0) as ctx, pb.Grid(ctx, p.grid, p.atoms) as g:
        got = g.export("ghost")
    assert want.min() < 1e-300 and want.max() > 1e-3
    # kappa r from the value itself: |ln| of a term is kappa r + ln(eps r / q), ln at most 14
    kr = np.maximum(0.0, -np.log(np.maximum(want, 5e-324)))
    tol = 2 * (9 + 2 * kr) * 2.0 ** -53
    assert np.all(np.abs(got - want) <= tol * np.abs(want) + 1e-290)
