"""NaN, infinities and non-physical states at precisions 64 and 48.

A row that cannot be evaluated (negative pressure, a NaN or an infinity, a
momentum beyond FP32's range) gives non-finite results wherever FP64 arithmetic
throughout gives them (fdu_residual_noalloc, or the same state in density units
outside the double words' window), and every other row its FP64 value: the
double words may not turn it into an ordinary number.  Tolerance on the finite
rows: the FP64 parity bound 1e-12 of the residual (1e-11 of a step's increment).
"""
import numpy as np
import pytest

from paper_2102_12933_gb300 import fdu, inputs

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

V = 137  # the vertex that is spoilt
ROWS = {
    "negative pressure": (1.0, 3.0, 0.0, 1.0),
    "nan momentum": (1.0, np.nan, 0.0, 2.0),
    "infinite momentum": (1.0, 0.0, -np.inf, 2.0),
    "huge momentum": (1.0, 1e200, 0.0, 2.0),
    "momentum beyond fp32": (1.0, 0.0, 1e60, 2.0),
    "negative energy": (1.0, 0.1, 0.0, -1.0),
    "nan density": (np.nan, 0.1, 0.0, 2.0),
    "infinite energy": (1.0, 0.1, 0.0, np.inf),
}


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _same(got, want, tol):
    """The same entries are finite, and those agree."""
    ok = np.isfinite(want)
    assert np.array_equal(np.isfinite(got), ok)
    assert _rel(got[ok], want[ok]) <= tol


def _mesh(n=24, **kw):
    m, w = inputs.vortex_case(n, seed=31)
    return fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, **kw), m, w


@pytest.mark.parametrize("row", ROWS)
@pytest.mark.parametrize("n", [24, 120])
def test_residual_rows(row, n):
    M, m, w = _mesh(n)
    w[V] = ROWS[row]
    t = torch.tensor(w, device="cuda")
    want, got = torch.empty_like(t), torch.empty_like(t)
    M.residual_noalloc(t, want)
    fallbacks = M.fallback_count(reset=True)
    M.set_state(t)
    M.residual(64, out=got)
    assert M.fallback_count() == fallbacks
    _same(got.cpu().numpy(), want.cpu().numpy(), 1e-12)


@pytest.mark.parametrize("row", ["nan momentum", "nan density"])
def test_precision_48_rows(row):
    M, m, w = _mesh()
    w[V] = ROWS[row]
    t = torch.tensor(w, device="cuda")
    want, got = torch.empty_like(t), torch.empty_like(t)
    M.residual_noalloc(t, want)
    fallbacks = M.fallback_count(reset=True)
    M.set_state(t)
    M.residual(48, out=got)
    assert M.fallback_count() == fallbacks
    _same(got.cpu().numpy(), want.cpu().numpy(), 1e-12)


@pytest.mark.parametrize("precision", [64, 48])
def test_stage_that_loses_its_pressure(precision):
    """A step far beyond the CFL bound at one vertex: its first stage has
    negative pressure, so the later stages are non-finite around it.  The same
    step in density units of 2^40 runs in FP64 throughout."""
    s = 2.0 ** 40
    m, w = inputs.vortex_case(24, seed=31)
    w[V, 3] *= 40.0
    out = []
    for scale, p in ((1.0, precision), (s, 64)):
        M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, weno_eps=1e-40 * scale * scale)
        M.set_state(w * scale)
        M.rk_step(M.max_dt(6.0), p)
        out.append(M.get_state() / scale)
    assert not np.isfinite(out[1]).all() and np.isfinite(out[1]).any()
    ok = np.isfinite(out[1])
    assert np.array_equal(np.isfinite(out[0]), ok)


@pytest.mark.parametrize("row", ROWS)
def test_vjp_rows(row):
    """Against the same state in density units of 2^30, which FP64 takes."""
    s = 2.0 ** 30
    m, w = inputs.vortex_case(24, seed=31)
    w[V] = ROWS[row]
    lam = torch.tensor(np.random.default_rng(1).standard_normal(w.shape), device="cuda")
    out = []
    for scale in (1.0, s):
        M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, weno_eps=1e-6 * scale * scale)
        M.set_state(torch.tensor(w * scale, device="cuda"))
        g = torch.empty_like(lam)
        M.residual_vjp(lam, out=g)
        out.append(g.cpu().numpy())
    _same(out[0], out[1], 1e-10)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_precision_48_cotangent(value):
    M, m, w = _mesh(weno_eps=1e-6)
    lam = np.random.default_rng(1).standard_normal(w.shape)
    lam[V, 2] = value
    M.set_state(w)
    out = []
    for p in (64, 48):
        M.set_adjoint_precision(p)
        out.append(M.residual_vjp(lam))
    assert not np.isfinite(out[0]).all()
    _same(out[1], out[0], 1e-10)


def test_split():
    x = np.array([np.nan, np.inf, -np.inf, 1e300, -1e39, 2.0 ** 128, -np.nan])
    assert not np.isfinite(fdu.check_dw("split", x)).any()
    big = np.array([2.0 ** 127, -3.4e38, 1e38])
    assert np.all(np.abs(fdu.check_dw("split", big) - big) <= 2.0 ** -47 * np.abs(big))
