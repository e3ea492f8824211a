"""FP32 stage with diffusion and a velocity along one axis only: along the others a
point reads the Laplacian's neighbours and nothing more.  A NaN shows what is read;
both stage kernels must leave the same points finite."""
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


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("order", [2, 4])
def test_nan_reach(mr, axis, order):
    nb, nt, at = 16, (2, 1, 1), (7, 8, 6)  # x, y, z of the NaN in the first leaf
    lev, anc = I.uniform_leaves(nt, 0)
    rng = np.random.default_rng(order)
    phi = rng.uniform(-1, 1, (2, nb, nb, nb)).astype(np.float32)
    phi[0, at[2], at[1], at[0]] = np.nan
    u = [0.0, 0.0, 0.0]
    u[axis] = 0.5
    masks = []
    for kernel in (1, 2):
        g = mr.Grid(nt, 0.5, nb, 0, 0, 2, 2, lev, anc, precision=mr.F32, nfields=2)
        g.set_stage_kernel(kernel)
        g.set_diffusion(0.01, order)
        g.field_copy_in(0, phi)
        g.rhs_advect(0, u, 1, mr.WENOZ5)
        masks.append(np.isnan(g.field_copy_out(1)))
    want = np.zeros_like(masks[0])
    for d in range(3):
        # a cell reads its own column from 3 behind to 2 ahead of it
        reach = range(-2, 4) if d == axis else range(-order // 2, order // 2 + 1)
        for k in reach:
            p = list(at)
            p[d] += k
            want[0, p[2], p[1], p[0]] = True
    assert np.array_equal(masks[0], want) and np.array_equal(masks[1], want)
