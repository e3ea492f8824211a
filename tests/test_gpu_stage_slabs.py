"""FP32 stage kernel on block sizes that its slabs cut unevenly, next to same-level,
coarser and finer leaves (for N.0 the finer leaves are read directly, and a slab
may end on either side of the boundary between two of them), in both walk
directions along z.  Bound: 1e-5 of the field maximum against the FP64 oracle, the
FP32 tolerance of the other stage tests."""
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


@pytest.mark.parametrize("nb,N,Nt", [(8, 2, 0), (10, 2, 2), (14, 4, 0), (18, 4, 2), (20, 2, 0), (22, 6, 2), (26, 4, 0)])
@pytest.mark.parametrize("mode", ["up", "down", "fields", "diffusion"])
def test_slabs_match_oracle(mr, oracle_mod, nb, N, Nt, mode):
    O, (nt, tl) = oracle_mod, ((2, 2, 2), 0.5)
    lev, anc = I.tree_config1()
    vel, diff = mode == "fields", 2 if mode == "diffusion" else 0
    g = mr.Grid(nt, tl, nb, 0, 1, N, Nt, lev, anc, precision=mr.F32, nfields=4 if vel else 1, velocity=vel)
    g.set_stage_kernel(1)
    lev, anc, _ = g.leaves()
    og = O.Grid(nt, tl, nb, N, Nt, 0, 1, lev, anc)
    xyz = I.point_coords(nt, tl, nb, lev, anc)
    phi = I.gaussian_images(xyz, (0.45, 0.5, 0.55), 0.12, nimg=1).astype(np.float32)
    g.field_copy_in(0, phi)
    h, ref = tl / (nb * 2), phi.astype(np.float64)
    if vel:
        w = 2 * np.pi
        v = [np.sin(w * xyz[d] + d) * np.cos(w * xyz[(d + 1) % 3]) for d in range(3)]
        v = [x.astype(np.float32) for x in v]
        for d in range(3):
            g.field_copy_in(1 + d, v[d])
        pads = [O.ghost_fill(og, O.ghost_fill(og, x.astype(np.float64), 3)[1], 3)[0] for x in v]
        g.step_vel(0, 0.2 * h, (1, 2, 3), mr.WENOZ5)
        ref = O.rk3_step_velpad(og, ref, pads, 0.2 * h, O.WENOZ5)
    else:
        u = (0.8, -0.6, 0.5 if mode == "up" else -0.5)
        dt = 0.2 * h
        if diff:
            g.set_diffusion(0.01, diff)
            dt = min(dt, 0.1 * h * h / 0.01)
        g.step(0, dt, u, mr.WENOZ5)
        ref = (O.rk3_step_diff(og, ref, dt, O.WENOZ5, u, 0.01, diff) if diff
               else O.rk3_step(og, ref, dt, O.WENOZ5, u))
    assert np.abs(g.field_copy_out(0) - ref).max() <= 1e-5 * np.abs(ref).max()
