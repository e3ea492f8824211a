"""Calls on the largest blocks of FP32 grids: what is refused, with which code, and
the block norms of the largest accepted one (float pairs, 41^3 extended regions); and
the norms of FP64 grids of many leaves.  Norms within 1e-12 of the field maximum, as
in test_gpu_adapt_tiles.py."""
import numpy as np
import pytest

from paper_2112_07537_gb300 import inputs as I

pytestmark = pytest.mark.gpu
INVALID, CUDA, UNSUPPORTED = -1, -3, -5


@pytest.fixture(scope="module")
def mr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_07537_gb300 import build, mrgb
    build.build()
    return mrgb


def _grid(mr, nb, N, Nt):
    lev, anc = I.uniform_leaves((2, 1, 1), 0)
    lev, anc = I.refine_leaves(lev, anc, anc[:, 0] == 0)
    return mr.Grid((2, 1, 1), 0.5, nb, 0, 1, N, Nt, lev, anc, precision=mr.F32, nfields=2)


def _code(mr, call, *args):
    with pytest.raises(mr.MRError) as e:
        call(*args)
    return e.value.code


@pytest.mark.parametrize("nb", [28, 32])
def test_stage_refusals(mr, nb):
    g = _grid(mr, nb, 4, 2)
    g.field_copy_in(0, np.ones((g.nleaf, nb, nb, nb), np.float32))
    assert _code(mr, g.step, 0, 1e-3, (1.0, 0.5, 0.0), 3) == INVALID  # no such scheme
    assert _code(mr, g.step, 0, 1e-3, (1.0, 0.5, 0.0), mr.WENOZ5) == CUDA
    g.sync()


def test_largest_float_pair_norms(mr, oracle_mod):
    import torch
    nb = 32
    g = _grid(mr, nb, 6, 0)
    lev, anc, _ = g.leaves()
    phi = np.random.default_rng(1).uniform(-1, 1, (g.nleaf, nb, nb, nb)).astype(np.float32)
    g.field_copy_in(0, phi)
    md = torch.empty(g.nleaf, dtype=torch.float64, device="cuda")
    g.criterion(0, md)
    g.sync()
    og = oracle_mod.Grid((2, 1, 1), 0.5, nb, 6, 0, 0, 1, lev, anc)
    ref = oracle_mod.block_maxdet(og, phi.astype(np.float64))
    assert np.abs(md.cpu().numpy() - ref).max() <= 1e-12 * np.abs(phi).max()
    big = _grid(mr, nb, 6, 2)
    big.field_copy_in(0, phi)
    assert _code(mr, big.criterion, 0, md) == UNSUPPORTED


@pytest.mark.parametrize("nb,N,Nt,n", [(8, 2, 2, 6), (18, 4, 0, 6), (26, 4, 2, 5), (32, 2, 0, 5)])
def test_fp64_norms_of_many_leaves(mr, oracle_mod, nb, N, Nt, n):
    """FP64 grids of more tiles than SMs, among them regions of more points per plane
    than a CTA has threads."""
    import torch
    nt = (n, n, n)
    lev, anc = I.uniform_leaves(nt, 0)
    lev, anc = I.refine_leaves(lev, anc, np.all(anc == 0, axis=1))
    g = mr.Grid(nt, 0.5, nb, 0, 1, N, Nt, lev, anc, precision=mr.F64)
    lev, anc, _ = g.leaves()
    phi = np.random.default_rng(nb).uniform(-1, 1, (g.nleaf, nb, nb, nb))
    g.field_copy_in(0, phi)
    md = torch.empty(g.nleaf, dtype=torch.float64, device="cuda")
    g.criterion(0, md)
    g.sync()
    ref = oracle_mod.block_maxdet(oracle_mod.Grid(nt, 0.5, nb, N, Nt, 0, 1, lev, anc), phi)
    assert np.abs(md.cpu().numpy() - ref).max() <= 1e-12 * np.abs(phi).max()
