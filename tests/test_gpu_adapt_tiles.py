"""Criterion column tiles, child / parent interpolation and the update boxes at
block sizes where tiles, runs and parities end differently.

Every leaf holds noise and one spike at a point of its own, so the block norm
comes from another point (edges and corners of the tiles included) of each
block.  The bounds are those of the neighbouring adaptation tests: 1e-12 of the
field maximum for FP64 results (sums of products of order 1 in another order)
and for the block norms, 2e-6 of it for FP32 fields (FP32 filters, a few dozen
roundings of 6e-8)."""
import numpy as np
import pytest

from paper_2112_07537_gb300 import inputs as I

pytestmark = pytest.mark.gpu
NT, TL = (5, 3, 3), 0.25


@pytest.fixture(scope="module")
def mr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_07537_gb300 import build, mrgb
    build.build()
    return mrgb


def _tree():
    lev, anc = I.uniform_leaves(NT, 0)
    hit = (anc[:, 0] >= 1) & (anc[:, 0] <= 3) & np.all(anc[:, 1:] <= 1, axis=1)
    lev, anc = I.refine_leaves(lev, anc, hit)
    return I.balance(NT, lev, anc)


def _field(nb, lev, anc, prec, seed):
    """Noise of 1e-2 in the trees x = 0..2 (those at x = 1 coarsen, their fine
    neighbours at x = 2 touch the noise of 1 beyond and stay), a spike of 100 in
    one coarse leaf."""
    rng = np.random.default_rng(seed)
    phi = rng.uniform(-1, 1, (len(lev), nb, nb, nb)) * np.where(anc[:, 0] >> lev <= 2, 1e-2, 1.0)[:, None, None, None]
    phi[np.flatnonzero((lev == 0) & (anc[:, 0] == 4) & (anc[:, 1] == 2))[-1], nb // 2, nb - 1, 1] = 100.0
    return phi.astype(np.float32) if prec else phi


def _pair(mr, O, nb, N, Nt, prec):
    lev, anc = _tree()
    g = mr.Grid(NT, TL, nb, 0, 3, N, Nt, lev, anc, precision=mr.F32 if prec else mr.F64, nfields=2,
                capacity=2000)
    lev, anc, _ = g.leaves()
    return g, O.Grid(NT, TL, nb, N, Nt, 0, 3, lev, anc)


# (nb, N, Nt, prec): FP32 32^3 blocks with 6.2 exceed what the criterion takes
CRIT = [(nb, N, Nt, p) for nb, N, Nt in [(8, 2, 2), (10, 4, 0), (14, 4, 2), (18, 2, 0), (20, 4, 2), (26, 6, 2),
                                         (30, 4, 2), (32, 2, 2), (32, 6, 0)] for p in (0, 1)
        if not (p and (nb, N, Nt) == (32, 6, 0))]


@pytest.mark.parametrize("nb,N,Nt,prec", CRIT)
def test_criterion_tiles(mr, oracle_mod, nb, N, Nt, prec):
    import torch
    g, og = _pair(mr, oracle_mod, nb, N, Nt, prec)
    rng = np.random.default_rng(nb + N)
    phi = 0.1 * rng.uniform(-1, 1, (g.nleaf, nb, nb, nb))
    at = rng.integers(0, nb, (g.nleaf, 3))
    at[:8] = np.array([[x, y, z] for x in (0, nb - 1) for y in (0, nb - 1) for z in (0, nb - 1)])
    phi[np.arange(g.nleaf), at[:, 2], at[:, 1], at[:, 0]] = rng.uniform(1, 2, g.nleaf)
    phi = phi.astype(np.float32) if prec else phi
    g.field_copy_in(0, phi)
    md = torch.empty(g.nleaf, dtype=torch.float64, device="cuda")
    g.criterion(0, md)
    g.sync()
    ref = oracle_mod.block_maxdet(og, phi.astype(np.float64))
    assert np.abs(md.cpu().numpy() - ref).max() <= 1e-12 * np.abs(phi).max()


@pytest.mark.parametrize("nb,N,Nt,prec", [(nb, N, Nt, p) for nb, N, Nt in [(8, 2, 2), (10, 4, 0), (14, 4, 2), (18, 2, 0),
                                                                           (20, 4, 2)] for p in (0, 1)] + [(22, 6, 2, 1)])
def test_adapt_iteration_block_sizes(mr, oracle_mod, nb, N, Nt, prec):
    """Refined, coarsened, updated and copied blocks of two fields."""
    O = oracle_mod
    g, og = _pair(mr, O, nb, N, Nt, prec)
    phis = [_field(nb, og.lev, og.anc, prec, s) for s in (1, 2)]
    for f, p in enumerate(phis):
        g.field_copy_in(f, p)
    p64 = [p.astype(np.float64) for p in phis]
    md, (er, ec) = O.block_maxdet(og, p64[0]), (30.0, 0.2)
    assert min(np.abs(md - er).min(), np.abs(md - ec).min()) > 1e-6
    og2, outs, _, onch, _, st = O.adapt_iter_fields(og, p64, er, ec)
    assert (st == 1).any() and (st == -1).any() and (st[og.lev > 0] == 0).any()
    assert g.adapt_iter(0, er, ec) == onch
    lev, anc, _ = g.leaves()
    assert np.array_equal(lev, og2.lev) and np.array_equal(anc, og2.anc)
    for f, ref in enumerate(outs):
        err = np.abs(g.field_copy_out(f).astype(np.float64) - ref.reshape(len(lev), nb, nb, nb)).max()
        assert err <= (2e-6 if prec else 1e-12) * np.abs(ref).max()
