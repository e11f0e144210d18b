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
