"""The FP64-state divergence with one, two and four lanes to a vertex.

The number of lanes follows the vertex count (up to 12,288: four, up to 57,344:
two); the lattices lie on both sides of each line, with counts that leave every
kind of warp remainder.  The vertices checked are sampled, the oracle serves
those alone; tolerance: the FP64 parity bound 1e-12."""
import numpy as np
import pytest

import oracle
from paper_2102_12933_gb300 import fdu, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9, 25, 110, 111, 239, 240])
@pytest.mark.parametrize("precision", [64, 48])
def test_residual_at_the_lane_counts(n, precision):
    m, w = inputs.vortex_case(n, seed=70 + n)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly)
    pick = np.unique(np.random.default_rng(n).integers(0, m.nv, 600))
    pick = np.union1d(pick, [0, m.nv - 1])
    mask = np.zeros(m.nv, np.uint8)
    mask[pick] = 1
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)
    M.set_state(w)
    want, got = om.residual(w, mask=mask)[pick], M.residual(precision)[pick]
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
