"""The double-word edge flux of precisions 64 and 48 where its dispatch turns.

The edge kernel gives each thread one edge in blocks of 128 and pairs the left
and right states in the lanes of packed instructions; the meshes below have
edge counts that leave every kind of remainder (3 n^2 edges on an n x n torus),
from the smallest lattice the stencils fit on.  Precision 64 leaves the double
words per stage (a density or energy outside 2^-24 .. 2^24 anywhere) and per
edge (Mach number above 3.9); the states below lie on both sides of each line.
Tolerance: the FP64 parity bound 1e-12 of the path; where the flow is
hypersonic the pressure is a small difference, p / (rho E) ~ 2.5 / M^2, which
multiplies the rounding of either side's pressure by M^2: 1e-12 M^2 / 10.
"""
import numpy as np
import pytest

import oracle
from paper_2102_12933_gb300 import fdu, inputs

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("precision", [64, 48])
@pytest.mark.parametrize("n", [7, 11, 13, 16, 21, 33])
def test_residual_matches_oracle(n, precision):
    m, w = inputs.vortex_case(n, seed=40 + n)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)
    M.set_state(w)
    assert _rel(M.residual(precision), om.residual(w)) <= 1e-12


@pytest.mark.parametrize("rho,vel", [(2.0 ** 20, 1.0), (2.0 ** -20, 1.0), (2.0 ** 25, 1.0), (2.0 ** -26, 1.0),
                                     (2.0 ** 60, 1.0), (1.0, 2.0 ** 9), (1.0, 2.0 ** -10), (1.0, 2.0 ** 30),
                                     (2.0 ** -100, 2.0 ** 30)])
def test_scaled_states_take_the_same_steps(rho, vel):
    """The Euler equations in other units: densities times rho, velocities
    times vel (powers of two, exact), time steps divided by vel.  Inside the
    window the double-word path serves them, outside the FP64 one; both give
    the unit-scale step to rounding."""
    m, w = inputs.vortex_case(21, seed=5)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly)
    scale = np.array([rho, rho * vel, rho * vel, rho * vel * vel])
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, weno_eps=1e-300)
    M.set_state(w * scale)
    L = om.residual(w, eps=1e-300)
    assert _rel(M.residual(64) / (scale * vel), L) <= 1e-12
    dt = om.max_dt(w, 0.4)
    want = w
    for _ in range(3):
        M.rk_step(dt / vel, 64)
        want = om.rk3_step(want, dt, eps=1e-300)
    assert _rel(M.get_state() / scale - w, want - w) <= 1e-11


@pytest.mark.parametrize("mach", [3.0, 5.0, 20.0])
def test_fast_flow_matches_oracle(mach):
    m, w = inputs.vortex_case(21, seed=6)
    x, y = 2 * np.pi * m.xy.T / 10
    rho, p = 1 + 0.2 * np.sin(x) * np.cos(y), 1 / 1.4 * (1 + 0.2 * np.cos(x - 1))
    w = inputs.primitive_to_conservative(rho, mach * (1 + 0.05 * np.sin(y)), 0.3 * mach + 0.1 * np.cos(x), p)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)
    M.set_state(w)
    assert _rel(M.residual(64), om.residual(w)) <= 1e-12 * max(1.0, mach * mach / 10)


def test_one_vertex_outside_the_window():
    """A single state outside the window sends the stage to FP64; the next
    state, inside it, comes back to the double words."""
    m, w = inputs.vortex_case(16, seed=8)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)
    w = w * 2.0 ** 22  # energies up to 3.6 2^22, below 2^24
    v = w.copy()
    v[37] *= 1.5  # 5.2 2^22
    for state in (v, w, v):
        M.set_state(state)
        assert _rel(M.residual(64), om.residual(state)) <= 1e-12
