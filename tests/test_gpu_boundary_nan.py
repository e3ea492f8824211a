"""A NaN in the field of a grid with physical boundaries is data, not a balance
error: the ghost fill passes it on to the ghosts of a finer neighbour and mr_sync
reports nothing."""
import numpy as np
import pytest

from paper_2112_07537_gb300 import inputs as I
from test_gpu_boundary import mr  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,fp64", [(0, False), (0, True), (1, False)])
@pytest.mark.parametrize("bounded", [(1, 1, 1), (1, 0, 0)])
def test_nan_is_no_balance_error(mr, prec, fp64, bounded):  # noqa: F811
    import torch
    nb, G = 16, 3
    lev, anc = I.tree_config1()
    g = mr.Grid((2, 2, 2), 0.5, nb, 0, 1, 4, 2, lev, anc, precision=prec, bounded=bounded)
    lev, anc, _ = g.leaves()
    f = np.ones((len(lev), nb, nb, nb), g.np_dtype)
    coarse = np.flatnonzero((lev == 0) & np.all(anc == (1, 0, 0), axis=1))[0]  # next to the refined tree (0, 0, 0)
    f[coarse, 2, 2, 0] = np.nan
    g.field_copy_in(0, f)
    W = nb + 2 * G
    pad = torch.empty((len(lev), W, W, W), dtype=torch.float64 if fp64 or prec else torch.float32, device="cuda")
    (g.ghost_fill64 if fp64 else g.ghost_fill)(0, G, pad)
    g.sync()
    nan = torch.isnan(pad).flatten(1).any(1).cpu().numpy()
    assert nan[coarse] and nan[lev == 1].any()
