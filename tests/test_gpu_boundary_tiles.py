"""Ghost fills next to physical boundaries against the oracle over the pre-pass's
forms: whole boxes of refinement sums, boxes cut into chunks (FP64 blocks at the
adaptation shell, where the chunk must hold the polynomial's nodes), the
smallest and large blocks, and FP64 blocks of an FP32 field (point by point).
Tolerances as in test_gpu_boundary.py (the conditioning of the boundary
polynomials)."""
import numpy as np
import pytest

from test_gpu_boundary import _field, _grids, _tol
from test_gpu_boundary import mr  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nb,N,Nt,G,bc", [
    (1, 8, 4, 0, 3, 0),    # smallest block
    (1, 20, 2, 2, 3, 1),
    (0, 16, 4, 2, 3, 0),
    (1, 24, 6, 2, 11, 2),  # FP64 at the adaptation shell
    (1, 28, 6, 2, 11, 0),
])
def test_bounded_ghosts_by_tile(mr, oracle_mod, prec, nb, N, Nt, G, bc):  # noqa: F811
    import torch
    bounded = (1, 1, 1) if N < 6 else (1, 0, 0)
    g, og = _grids(mr, oracle_mod, N, Nt, nb, prec, bounded, bc)
    f = _field(og, nb).astype(np.float64 if prec else np.float32)
    ref_pad, ref_sub = oracle_mod.ghost_fill(og, f.astype(np.float64), G)
    g.field_copy_in(0, f)
    W = nb + 2 * G
    pad = torch.empty((g.nleaf, W, W, W), dtype=torch.float64 if prec else torch.float32, device="cuda")
    g.ghost_fill(0, G, pad)
    g.sync()
    scale = np.abs(ref_pad).max()
    assert np.abs(pad.cpu().numpy() - ref_pad).max() <= _tol(N, G, sum(bounded), prec) * scale
    assert np.abs(g.field_copy_out(0) - ref_sub).max() <= (1e-12 if prec else 1e-5) * scale


@pytest.mark.parametrize("nb,N,Nt", [(16, 4, 2), (20, 6, 0)])
def test_bounded_fp64_ghosts_of_fp32_field(mr, oracle_mod, nb, N, Nt):  # noqa: F811
    import torch
    g, og = _grids(mr, oracle_mod, N, Nt, nb, 0, (1, 0, 0), 0)
    f = _field(og, nb).astype(np.float32)
    G = oracle_mod.adapt_shell(N, Nt)
    ref_pad, _ = oracle_mod.ghost_fill(og, f.astype(np.float64), G)
    g.field_copy_in(0, f)
    W = nb + 2 * G
    pad = torch.empty((g.nleaf, W, W, W), dtype=torch.float64, device="cuda")
    g.ghost_fill64(0, G, pad)
    g.sync()
    assert np.abs(pad.cpu().numpy() - ref_pad).max() <= _tol(N, G, 1, 1) * np.abs(ref_pad).max()
