"""The range flags of precision 64 describe the state, not the calls before.

A state outside the double words' window (density or energy outside 2^-24 ..
2^24) is evaluated in FP64 throughout.  fdu_rk_step_vjp recomputes two of the
three stages and leaves the state in place, so the next call has to find that
state's flags again: the same bits before and after.
"""
import numpy as np
import pytest

from paper_2102_12933_gb300 import fdu, inputs

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("adjoint", [64, 48])
@pytest.mark.parametrize("s", [1.0, 2.0 ** 60, 2.0 ** -60])
def test_step_vjp_leaves_the_flags_of_its_state(s, adjoint):
    m, w = inputs.vortex_case(21, seed=5)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, weno_eps=1e-300)
    M.set_state(w * s)
    dt = M.max_dt(0.4)
    lam = np.random.default_rng(3).standard_normal(w.shape)
    first = M.residual(64)
    M.rk_step(dt, 64)
    stepped = M.get_state()
    M.set_state(w * s)
    M.set_adjoint_precision(adjoint)
    grads = []
    for _ in range(2):
        grads.append(M.rk_step_vjp(dt, lam))
        assert np.array_equal(M.get_state(), w * s)
        assert np.array_equal(M.residual(64), first)
    assert np.array_equal(grads[0], grads[1])
    M.rk_step_vjp(dt, lam)
    M.rk_step(dt, 64)
    assert np.array_equal(M.get_state(), stepped)


@pytest.mark.parametrize("n", [16, 110, 111, 240])
def test_wide_state_over_the_lanes_of_a_vertex(n):
    """FP64 throughout with four (to 12,288 vertices), two (to 57,344) and one
    lane to a vertex: fdu_residual_noalloc to 1e-13 (the same sums, without
    the vertices' Roe records), and a step in density units of 2^40 to the parity bound
    1e-11 of the increment."""
    s = 2.0 ** 40
    m, w = inputs.vortex_case(n, seed=n)
    M = fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly, weno_eps=1e-300)
    t = torch.tensor(w * s, device="cuda")
    want, got = torch.empty_like(t), torch.empty_like(t)
    M.residual_noalloc(t, want)
    M.set_state(t)
    M.residual(64, out=got)
    assert float(torch.linalg.norm(got - want) / torch.linalg.norm(want)) <= 1e-13
    dt = M.max_dt(0.4)
    M.rk_step(dt, 64)
    wide = M.get_state() / s
    M.set_state(w)
    M.rk_step(dt, 64)
    one = M.get_state()
    assert np.linalg.norm(wide - one) <= 1e-11 * np.linalg.norm(one - w)


@pytest.mark.parametrize("sizes", [(16, 23, 29), (60, 90, 100), (150, 160, 170)])
@pytest.mark.parametrize("spoilt", [0, 1, 2])
def test_meshes_of_a_batch_keep_to_themselves(sizes, spoilt):
    """One mesh of a batch outside the window (in density units of 2^40): it takes
    the bits that it has when all of them are, and the others those that they
    have when none is, in residuals (four, two and one lanes to a vertex) and in
    persistent steps."""
    cases = [inputs.vortex_case(n, seed=n, beta=3.0) for n in sizes]
    B = fdu.Batch([(m.xy, m.tri) for m, _ in cases], L=10.0, weno_eps=1e-300)
    s = 2.0 ** 40
    scale = {"none": [1.0] * 3, "all": [s] * 3, "one": [s if i == spoilt else 1.0 for i in range(3)]}
    out = {}
    for k, f in scale.items():
        B.set_state(np.concatenate([w * a for (_, w), a in zip(cases, f)]))
        B.set_dt(B.batch_max_dt(0.4))
        r = B.residual(64)
        B.batch_rk_steps(2, 64)
        p = B.get_state()
        B.rk_step(1e-3, 64)
        out[k] = (r, p, B.get_state())
    for i in range(3):
        rows = slice(B.offsets[i], B.offsets[i + 1])
        for got, want in zip(out["one"], out["all" if i == spoilt else "none"]):
            assert np.array_equal(got[rows], want[rows])
