"""The precision-48 edge flux at sizes around its block and warp edges.

The edge kernel gives each thread one edge in blocks of 128 and pairs the left
and right states in the lanes of packed instructions; the meshes below have
edge counts that leave every kind of remainder (3 n^2 edges on an n x n torus),
from the smallest lattice the stencils fit on.  Tolerance: the FP64 parity
bound 1e-12 of the path (FP64 state terms, increments to about 2^-46).
"""
import numpy as np
import pytest

import oracle
from paper_2102_12933_gb300 import fdu, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [48])
@pytest.mark.parametrize("n", [7, 11, 13, 16, 21, 33])
def test_residual_matches_oracle(n, precision):
    m, w = inputs.vortex_case(n, seed=40 + n)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)
    M.set_state(w)
    want = om.residual(w)
    got = M.residual(precision)
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
