"""The FP32 divergence over tiles of 128 vertices staged in shared memory.

Sizes around the tile (128), slice (32) and group (4 entries) edges, ghost
layers, stencils of every size the options give, and a vertex order without
locality (shuffled ids, renumber = 0), where the tiles hold too many distinct
fluxes and the divergence gathers from global memory instead.  Tolerance: the
FP32 path's bound against the oracle, 1e-4 relative L2 of the residual."""
import numpy as np
import pytest

import oracle
from paper_2102_12933_gb300 import fdu, inputs

pytestmark = pytest.mark.gpu


def _check(m, w, **kw):
    degree = kw.get("lsq_degree", 2)
    om = oracle.OracleMesh(m.xy, m.tri, m.Lx, m.Ly, degree=degree, levels=kw.get("lsq_levels", 2), ghost=m.ghost_donor,
                           artificial=1 if isinstance(m.tri, tuple) else None)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, ghost_donor=m.ghost_donor, **kw)
    M.set_state(w)
    want, got = om.residual(w), M.residual(32)
    assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)
    dt = om.max_dt(w, 0.3)
    M.rk_step(dt, 32)
    w1 = om.rk3_step(w, dt)
    assert np.linalg.norm(M.get_state() - w1) <= 1e-5 * np.linalg.norm(w1)


@pytest.mark.parametrize("n", [7, 8, 11, 12, 16, 23, 32])
def test_sizes(n):
    _check(*inputs.vortex_case(n, seed=60 + n))


@pytest.mark.parametrize("degree,levels", [(1, 1), (1, 2), (3, 2), (5, 2)])
def test_stencil_sizes(degree, levels):
    _check(*inputs.vortex_case(19, seed=9, random_diagonals=False, jitter=0.05), lsq_degree=degree, lsq_levels=levels)


def test_ghost_layers():
    m, w = inputs.riemann_case(25, seed=4)
    w = w[np.where(m.ghost_donor < 0, np.arange(m.nv), m.ghost_donor)]
    _check(m, w)


def test_hybrid():
    m = inputs.hybrid_lattice(17, seed=2)
    _check(m, inputs.isentropic_vortex(m.xy))


@pytest.mark.parametrize("renumber", [0, 1])
def test_order_without_locality(renumber):
    m, w = inputs.vortex_case(64, seed=3)
    p, perm = inputs.permute_vertices(m, 1)
    _check(p, w[perm], renumber=renumber)


def test_nonfinite_flux_stays_in_its_stencils():
    """A NaN state reaches the residual of the vertices whose stencils hold it
    and of no others (padding entries repeat an entry of their own vertex)."""
    m, w = inputs.vortex_case(24, seed=5)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)
    import torch

    v = torch.tensor(w, device="cuda")
    v[100] = float("nan")
    M.set_state(v)
    out = torch.empty_like(v)
    M.residual(32, out=out)
    bad = ~np.isfinite(out.cpu().numpy()).all(1)
    M.residual(64, out=out)
    bad64 = ~np.isfinite(out.cpu().numpy()).all(1)
    assert bad.any() and not bad.all() and np.array_equal(bad, bad64)
