"""Precision 64 across steps of the state, against FP64 throughout.

A thin state formed from a dense one (density ratio r) costs the double words
log2 r of their 48 bits, and steps of more than a factor of two cost the VJP as
much, so such edges are taken in FP64.  Tolerance: FP64 is within 5e-14 of the
exact residual and within 7e-14 of the exact VJP on these states, and precision
64 is to be no further, so the two differ by at most 1e-13 and 1.4e-13; 2e-13.
"""
import numpy as np
import pytest

from paper_2102_12933_gb300 import fdu, inputs

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("ratio", [8, 1024, 4096])
def test_residual_across_density_steps(ratio):
    m = inputs.torus_lattice(48, seed=11)
    x = m.xy[:, 0]
    thin = np.where(np.abs(x - 5) < 2.5, 1.0, 1.0 / ratio)
    w = inputs.primitive_to_conservative(thin, np.where(x > 5, 1.0, -1.0), np.full(m.nv, 0.3), thin)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)
    M.set_state(w)
    t = torch.tensor(w, device="cuda")
    want = torch.empty_like(t)
    M.residual_noalloc(t, want)
    got, want = M.residual(64), want.cpu().numpy()
    scale = np.abs(want).max(axis=0)
    assert _rel(got / scale, want / scale) <= 2e-13


@pytest.mark.parametrize("ratio", [16, 64])
def test_vjp_across_steps(ratio):
    """FP64 throughout: the same state in density units of 2^30."""
    m = inputs.torus_lattice(48, seed=11)
    rng = np.random.default_rng(5)
    noise = lambda: 1 + 0.01 * rng.uniform(-1, 1, m.nv)  # noqa: E731
    thin = np.where(np.abs(m.xy[:, 0] - 5) < 2.5, 1.0, 1.0 / ratio)
    w = inputs.primitive_to_conservative(thin * noise(), 0.3 * noise(), 0.01 * noise(), thin * noise())
    lam = rng.standard_normal(w.shape)
    out = []
    for s in (1.0, 2.0 ** 30):
        M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, weno_eps=1e-6 * s * s)
        M.set_state(w * s)
        out.append(M.residual_vjp(lam))
    assert _rel(out[0], out[1]) <= 2e-13


@pytest.mark.parametrize("k,e", [(0, -60), (10, -90), (10, -100), (10, -110), (20, -110), (-10, -60), (-10, -100)])
def test_vjp_with_an_epsilon_below_the_noise_of_the_state(k, e):
    """A state with rounding noise, in units of density 2^k and velocity 2^-k, with
    epsilon = 2^e of the density squared: where noise (2^-106 of it) would pass
    for an indicator the derivative is FP64's, whatever the units.  Tolerance:
    the adjoint's bound 1e-10."""
    m = inputs.torus_lattice(32, seed=4)
    rng = np.random.default_rng(1)
    bump = 1 + 0.3 * np.exp(-4 * ((m.xy - 5) ** 2).sum(1))
    w = inputs.primitive_to_conservative(bump, 0.7 + 0 * bump, 0.3 + 0 * bump, bump / 1.4)
    w = w * (1 + 2.0 ** -52 * rng.integers(-3, 4, w.shape))
    lam = rng.standard_normal(w.shape)
    rho, vel = 2.0 ** k, 2.0 ** -k
    unit = np.array([rho, rho * vel, rho * vel, rho * vel * vel])
    out = []
    for s in (1.0, 2.0 ** 40):
        M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, weno_eps=rho * rho * s * s * 2.0 ** e)
        M.set_state(w * unit * s)
        out.append(M.residual_vjp(lam / unit) * unit)
    assert _rel(out[0], out[1]) <= 1e-10
