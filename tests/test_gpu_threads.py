"""Two host threads, each stepping and measuring a grid of its own on a stream of its
own: the grids differ in block size, so the same kernels are launched with different
amounts of shared memory at the same time.  Every call must succeed, and the fields
must be those of the same calls made one thread after the other, bit for bit."""
import threading

import numpy as np
import pytest

from paper_2112_07537_gb300 import inputs as I

pytestmark = pytest.mark.gpu
STEPS = 150


@pytest.fixture(scope="module")
def mr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_07537_gb300 import build, mrgb
    build.build()
    return mrgb


def _grid(mr, nb, prec, stream):
    import torch
    lev, anc = I.tree_config1()
    with torch.cuda.stream(stream):
        g = mr.Grid((2, 2, 2), 0.5, nb, 0, 1, 6, 0, lev, anc, precision=prec, nfields=2, stream=stream)
        lev, anc, _ = g.leaves()
        xyz = I.point_coords((2, 2, 2), 0.5, nb, lev, anc)
        phi = I.gaussian(xyz, (0.45, 0.5, 0.55), 0.12)
        g.field_copy_in(0, phi.astype(g.np_dtype))
        md = torch.empty(g.nleaf, dtype=torch.float64, device="cuda")
    return g, md


def _work(mr, g, md):
    for _ in range(STEPS):
        g.step(0, 1e-4, (0.8, -0.5, 0.3), mr.WENOZ5)
        g.criterion(0, md)
    g.sync()


@pytest.mark.parametrize("prec", [0, 1])
def test_two_threads_two_block_sizes(mr, prec):
    import torch
    sizes = (18, 32 if prec else 26)
    alone, err = [], []
    for nb in sizes:
        g, md = _grid(mr, nb, prec, torch.cuda.Stream())
        _work(mr, g, md)
        alone.append(g.field_copy_out(0))
    grids = [_grid(mr, nb, prec, torch.cuda.Stream()) for nb in sizes]

    def run(k):
        try:
            _work(mr, *grids[k])
        except mr.MRError as e:
            err.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not err, err
    for (g, _), ref in zip(grids, alone):
        assert np.array_equal(g.field_copy_out(0), ref)
