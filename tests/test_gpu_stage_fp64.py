"""The FP64 stage kernel against the oracle at the edges of its slabs and line
segments: block sizes whose z extent does not divide by the slab height, grids
from a few leaves (two-plane slabs, four-cell segments) to enough for full
slabs, and values that take the WENO-Z weights' quotient path (jumps, where
the cap acts; magnitudes whose products would overflow).

Tolerance: 1e-12 of the field maximum, as the other FP64 steps (about 1e3
operations per point and stage, each within 2^-53 of values no larger than a
few times the maximum: 1e3 * 1.1e-16 * 3 = 3e-13); the bare right-hand side at 1e-12
of its maximum likewise.  A jump is compared through the bare right-hand side
only: after one stage its symmetric profiles make tau = |beta_0 - beta_2| a
difference of equal values, and a step of the oracle itself then moves by 1e-5
when one velocity component changes by its last bit.
"""
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


CASES = [
    # nb, wavelet, trees, scheme, velocity fields, diffusion, values
    (8, (2, 0), (2, 2, 2), "WENOZ5", False, 0, "smooth"),
    (14, (4, 0), (2, 2, 2), "WENOZ5", True, 0, "smooth"),
    (18, (4, 2), (3, 2, 2), "CONS5", False, 4, "smooth"),
    (20, (2, 2), (4, 4, 3), "WENOZ5", False, 2, "smooth"),
    (10, (2, 2), (6, 5, 5), "CONS3", True, 0, "smooth"),
    (32, (4, 0), (1, 2, 2), "WENOZ5", False, 0, "smooth"),
    (16, (2, 0), (2, 2, 2), "WENOZ5", False, 0, "jump"),
    (16, (2, 0), (2, 2, 2), "WENOZ5", True, 0, "large"),
]


@pytest.mark.parametrize("nb,wav,nt,scheme,vel,diff,values", CASES)
def test_fp64_stage_matches_oracle(mr, oracle_mod, nb, wav, nt, scheme, vel, diff, values):
    O = oracle_mod
    tl = 1.0 / max(nt)
    lev, anc = I.uniform_leaves(nt, 0)
    lev, anc = I.refine_leaves(lev, anc, np.all(anc == 0, axis=1))
    lev, anc = I.balance(nt, lev, anc)
    g = mr.Grid(nt, tl, nb, 0, 1, wav[0], wav[1], lev, anc, precision=mr.F64, nfields=4 if vel else 2, velocity=vel)
    glev, ganc, _ = g.leaves()
    og = O.Grid(nt, tl, nb, wav[0], wav[1], 0, 1, glev, ganc)
    xyz = I.point_coords(nt, tl, nb, glev, ganc)
    ext = tuple(n * tl for n in nt)
    phi = I.gaussian(xyz, tuple(0.45 * e for e in ext), 0.15, ext)
    if values == "jump":
        phi = np.where(phi > 0.5, 1.0, 0.0)
    elif values == "large":
        phi = phi * 1e24
    g.field_copy_in(0, phi)
    h = tl / (nb * 2)
    dt, nu = 0.1 * h, 0.01 * h if diff else 0.0
    if diff:
        g.set_diffusion(nu, diff)
    sch = getattr(mr, scheme), getattr(O, scheme)
    if vel:
        v = [np.sin(2 * np.pi * xyz[(d + 1) % 3] / ext[(d + 1) % 3] + d) * (1.0 + 0 * xyz[0]) for d in range(3)]
        for d in range(3):
            g.field_copy_in(1 + d, np.ascontiguousarray(v[d]))
        vp = [O.ghost_fill(og, O.ghost_fill(og, np.ascontiguousarray(x), 3)[1], 3)[0] for x in v]
        g.step_vel(0, dt, (1, 2, 3), sch[0])
        ref = O.rk3_step_velpad(og, phi, vp, dt, sch[1])
    else:
        u = (0.8, -0.5, 0.0) if nb == 8 else (0.8, -0.5, 0.3)
        if values == "jump":
            g.rhs_advect(0, u, 1, sch[0])
            ref = O.rhs(og, O.ghost_fill(og, phi, 3)[0], 3, sch[1], u)
            assert np.abs(g.field_copy_out(1) - ref).max() <= 1e-12 * np.abs(ref).max()
            return
        g.step(0, dt, u, sch[0])
        ref = O.rk3_step_diff(og, phi, dt, sch[1], u, nu, diff) if diff else O.rk3_step(og, phi, dt, sch[1], u)
    got = g.field_copy_out(0)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
