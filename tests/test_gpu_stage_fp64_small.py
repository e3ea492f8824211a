"""FP64 stage kernel on fields far below the WENO-Z epsilon: every smoothness
term is 1e-30 there and the weights are the ideal ones, so step and right-hand
side scale with the field.  Bounds as in test_gpu_stage_fp64.py: 1e-12 of the
maximum of the oracle's result (at 1e-280 the smallest differences that count are
1e-292, above the subnormal range)."""
import numpy as np
import pytest

from paper_2112_07537_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_07537_gb300 import build, mrgb
    build.build()
    return mrgb


@pytest.mark.parametrize("scale", [1e-18, 1e-132, 1e-150, 1e-280])
@pytest.mark.parametrize("vel", [False, True])
def test_small_fields(mr, oracle_mod, vel, scale):
    O, nb, nt, tl = oracle_mod, 16, (2, 2, 2), 0.5
    lev, anc = I.uniform_leaves(nt, 0)
    lev, anc = I.refine_leaves(lev, anc, np.all(anc == 0, axis=1))
    g = mr.Grid(nt, tl, nb, 0, 1, 2, 0, lev, anc, precision=mr.F64, nfields=5, velocity=vel)
    glev, ganc, _ = g.leaves()
    og = O.Grid(nt, tl, nb, 2, 0, 0, 1, glev, ganc)
    xyz = I.point_coords(nt, tl, nb, glev, ganc)
    phi = I.gaussian(xyz, (0.45, 0.45, 0.45), 0.15) * scale
    dt = 0.1 * tl / (nb * 2)
    if vel:
        v = [np.ascontiguousarray(np.sin(2 * np.pi * xyz[(d + 1) % 3] + d) + 0 * xyz[0]) for d in range(3)]
        for d in range(3):
            g.field_copy_in(1 + d, v[d])
        vp = [O.ghost_fill(og, O.ghost_fill(og, x, 3)[1], 3)[0] for x in v]
        g.field_copy_in(0, phi)
        g.step_vel(0, dt, (1, 2, 3), mr.WENOZ5)
        pairs = [(g.field_copy_out(0), O.rk3_step_velpad(og, phi, vp, dt, O.WENOZ5))]
    else:
        u = (0.8, -0.5, 0.3)
        g.field_copy_in(0, phi)
        g.rhs_advect(0, u, 4, mr.WENOZ5)
        pairs = [(g.field_copy_out(4), O.rhs(og, O.ghost_fill(og, phi, 3)[0], 3, O.WENOZ5, u))]
        g.field_copy_in(0, phi)
        g.step(0, dt, u, mr.WENOZ5)
        pairs.append((g.field_copy_out(0), O.rk3_step(og, phi, dt, O.WENOZ5, u)))
    for got, ref in pairs:
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
