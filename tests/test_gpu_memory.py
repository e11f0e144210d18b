"""Device memory of a mesh: what it says it holds, and meshes that fit only
without the tables of the faster kernels.

Beside the tables that every path reads, a mesh keeps the double-word tables of
precisions 64 and 48 and the tiles of precision 32.  Where device memory ends
before those it is created without them: the same results to the parity bound
1e-12 in FP64, in FP32 no further from FP64 than twice what the tiles are (the
same terms in another order), and precision 48 is refused until there is room.
"""
import numpy as np
import pytest

from paper_2102_12933_gb300 import fdu, inputs

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

MB = 1 << 20


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def test_device_bytes_are_what_is_held():
    m, _ = inputs.vortex_case(24, seed=1)
    fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly).close()
    before = _free()
    meshes = [fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly) for _ in range(32)]
    held = before - _free()
    said = sum(M.info()["device_bytes"] for M in meshes)
    for M in meshes:
        M.close()
    assert said <= held <= 1.25 * said


@pytest.mark.parametrize("short", [24, 130])
def test_mesh_where_memory_ends(short):
    """Created with `short` MB less than a whole mesh takes: too little for the
    tiles, and for the double-word tables as well."""
    m, w = inputs.vortex_case(320, seed=2)
    make = lambda: fdu.Mesh(m.xy, m.tri, m.Lx, m.Ly)  # noqa: E731
    before = _free()
    M = make()
    M.set_state(w)
    want = {p: M.residual(p) for p in (64, 48, 32)}
    full = M.info()["device_bytes"]
    whole = before - _free()
    M.close()
    hog = torch.empty(_free() - whole + short * MB, dtype=torch.uint8, device="cuda")
    try:
        M = make()
        held = M.info()["device_bytes"]
        M.set_state(w)
        got = {p: M.residual(p) for p in (64, 32)}
        refused = False
        try:
            M.residual(48)
        except fdu.FduError:
            refused = True
        again = M.residual(64)
    finally:
        del hog
        _free()
    assert held < full - short * MB // 2
    assert _rel(got[64], want[64]) <= 1e-12
    assert _rel(got[32], want[64]) <= 2 * _rel(want[32], want[64])
    assert refused == (short > 100)
    assert np.array_equal(again, got[64])
    assert _rel(M.residual(48), want[48]) <= 1e-12
    M.rk_step(M.max_dt(0.2), 64)
    assert np.isfinite(M.get_state()).all()
    M.close()
