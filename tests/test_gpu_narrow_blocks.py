"""Ghost fills of blocks so narrow that the refinement of 6.x reads beyond the
neighbouring blocks, and of the next wider ones, on three levels of noise: FP64 and
FP32 against the oracle, within 1e-12 and 1e-5 of the field maximum (the tolerances of
the other ghost tests)."""
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


@pytest.mark.parametrize("nb,Nt", [(8, 0), (8, 2), (10, 0), (10, 2), (12, 2)])
@pytest.mark.parametrize("prec", [0, 1])
def test_narrow_blocks(mr, oracle_mod, nb, Nt, prec):
    import torch
    nt, tl, N, G = (3, 3, 2), 0.25, 6, 3
    lev, anc = I.uniform_leaves(nt, 0)
    lev, anc = I.refine_leaves(lev, anc, (anc[:, 0] == 0) & (anc[:, 1] <= 1))
    lev, anc = I.refine_leaves(lev, anc, (lev == 1) & np.all(anc == (1, 1, 1), axis=1))
    lev, anc = I.balance(nt, lev, anc)
    g = mr.Grid(nt, tl, nb, 0, 2, N, Nt, lev, anc, precision=prec, fixed_tree=True)
    lev, anc, _ = g.leaves()
    assert set(lev) == {0, 1, 2}
    phi = np.random.default_rng(nb).uniform(-1, 1, (len(lev), nb, nb, nb)).astype(g.np_dtype)
    g.field_copy_in(0, phi)
    pad = torch.empty((len(lev),) + (nb + 2 * G,) * 3, dtype=g.dtype, device="cuda")
    g.ghost_fill(0, G, pad)
    g.sync()
    ref, sub = oracle_mod.ghost_fill(oracle_mod.Grid(nt, tl, nb, N, Nt, 0, 2, lev, anc), phi.astype(np.float64), G)
    tol = (1e-12 if prec else 1e-5) * np.abs(ref).max()
    assert np.abs(pad.cpu().numpy() - ref).max() <= tol
    assert np.abs(g.field_copy_out(0) - sub).max() <= tol
