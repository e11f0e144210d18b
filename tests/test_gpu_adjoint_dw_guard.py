"""Where precision 64's edge VJP turns between double words and FP64.

In density units scaled by s (a power of two) the residual scales by s and its
VJP is the same numbers, with the WENO epsilon scaled by s^2.  Inside the
double words' window both scales run there, outside it the edges go to the FP64
kernel through the list; single edges do so where the flow is fast.  Cotangents
are linear, so scaling them by powers of two scales the result exactly.
Tolerance: the adjoint's bound 1e-10 (FP64 kernel: one-step reciprocals, 2^-40,
over sums of about ten terms)."""
import numpy as np
import pytest

from paper_2102_12933_gb300 import fdu, inputs

pytestmark = pytest.mark.gpu


def _case(n, mach=1.0):
    m, w = inputs.vortex_case(n, seed=80 + n)
    x, y = 2 * np.pi * m.xy.T / 10
    if mach > 1.0:
        w = inputs.primitive_to_conservative(1 + 0.2 * np.sin(x) * np.cos(y), mach * (1 + 0.5 * np.sin(y)), 0.3 + 0.1 * np.cos(x),
                                             1 / 1.4 * (1 + 0.2 * np.cos(x - 1)))
    for c in range(4):
        w[:, c] *= 1 + 0.02 * np.sin(x + 0.8 * c) * np.cos(y - 0.4 * c)
    return m, w


def _vjp(m, w, lam, eps, precision=64):
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, weno_eps=eps)
    M.set_adjoint_precision(precision)
    M.set_state(w)
    return M.residual_vjp(lam)


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n", [7, 11, 24])
@pytest.mark.parametrize("s", [2.0 ** 10, 2.0 ** 30, 2.0 ** -40])
def test_density_units(n, s):
    m, w = _case(n)
    lam = np.random.default_rng(n).standard_normal(w.shape)
    assert _rel(_vjp(m, w * s, lam, 1e-6 * s * s), _vjp(m, w, lam, 1e-6)) <= 1e-10


def test_fast_edges_and_small_epsilon():
    m, w = _case(24, mach=4.0)  # part of the edges beyond Mach 3.9
    lam = np.random.default_rng(1).standard_normal(w.shape)
    mixed = _vjp(m, w, lam, 1e-3)
    s = 2.0 ** 30  # all edges in FP64
    assert _rel(mixed, _vjp(m, w * s, lam, 1e-3 * s * s)) <= 1e-10


@pytest.mark.parametrize("k", [-900, -300, 300, 900])
@pytest.mark.parametrize("precision", [64, 48])
def test_cotangent_scale(k, precision):
    m, w = _case(11)
    lam = np.random.default_rng(2).standard_normal(w.shape)
    a, b = _vjp(m, w, lam, 1e-6, precision), _vjp(m, w, lam * 2.0 ** k, 1e-6, precision)
    assert _rel(b * 2.0 ** -k, a) <= 1e-13
