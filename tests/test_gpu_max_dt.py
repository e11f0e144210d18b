"""The CFL bound's FP32 screening: the bound is the FP64 minimum wherever it lies.

States whose smallest bound sits at one vertex, in ranges where FP32 resolves
the speed, where it does not (scales beyond its exponents, hypersonic flow), and
ties; odd vertex counts around the reduction's block (256).  Tolerance: 4 ulp of
the oracle's FP64 bound (one division and two square roots each side)."""
import numpy as np
import pytest

import oracle
from paper_2102_12933_gb300 import fdu, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 16, 17, 45])
@pytest.mark.parametrize("rho,vel", [(1.0, 1.0), (2.0 ** 40, 1.0), (2.0 ** -110, 1.0), (1.0, 2.0 ** 70), (1.0, 2.0 ** -80),
                                     (2.0 ** 120, 2.0 ** -90)])
def test_bound_is_the_minimum(n, rho, vel):
    m, w = inputs.vortex_case(n, seed=n)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)
    scale = np.array([rho, rho * vel, rho * vel, rho * vel * vel])
    rng = np.random.default_rng(n)
    for k in range(6):
        v = w.copy()
        i = int(rng.integers(m.nv))
        if k == 1:  # one fast vertex
            v[i] = [1.0, 3.0, 0.0, 2.5 + 4.5]
        elif k == 2:  # hypersonic everywhere, pressure 1e-6 of the energy
            v = inputs.primitive_to_conservative(np.ones(m.nv), 1.0 + 1e-9 * rng.standard_normal(m.nv), np.zeros(m.nv),
                                                 np.full(m.nv, 2e-7))
        elif k == 3:  # near ties
            v = np.tile(w[i], (m.nv, 1)) * (1 + 1e-13 * rng.standard_normal((m.nv, 1)))
        elif k == 4:  # one near-vacuum vertex
            v[i] = [1e-9, 1e-9, 0.0, 2.5e-3]
        elif k == 5:  # at rest
            v[:, 1:3] = 0.0
        M.set_state(v * scale)
        want = om.max_dt(v * scale, 0.5)
        assert abs(M.max_dt(0.5) - want) <= 4 * np.spacing(want)


def test_adaptive_steps_use_it():
    m, w = inputs.sod_case(30)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly, degree=5)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, lsq_degree=5)
    M.set_state(w)
    steps, t = M.advance(0.4, 1.0, 64, max_steps=11)
    want, u = 0.0, w
    for _ in range(11):
        dt = om.max_dt(u, 0.4)
        u, want = om.rk3_step(u, dt), want + dt
    assert steps == 11 and abs(t - want) <= 1e-12 * want
