"""What selects a kernel or its candidates is part of the autotuner's key: a choice
timed on a small grid, on a periodic one or without diffusion does not stand for a
large grid, for physical boundaries or for the stage kernel with diffusion."""
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


def _rows(mr, kernel):
    """{chosen: candidates} of the kernel's table rows, "k_prep ... -> 512 threads (512: .. ms, 256: .. ms)"."""
    rows = [ln for ln in mr.autotune_table() if ln.startswith(kernel)]
    return [[int(c.split(":")[0]) for c in ln[ln.rindex("(") + 1:ln.rindex(")")].split(",")] for ln in rows]


def test_key_separates_grids(mr):
    mr.autotune_clear()
    try:
        def grid(n, bounded):
            lev, anc = I.uniform_leaves((n, n, n), 0)
            g = mr.Grid((n, n, n), 1.0 / n, 16, 0, 0, 4, 2, lev, anc, precision=mr.F32, nfields=2, bounded=bounded)
            g.field_copy_in(0, np.ones((n ** 3, 16, 16, 16), np.float32))
            g.autotune(True)
            g.ghost_fill(0, 3)
            g.sync()
            return g

        small = grid(2, (0, 0, 0))
        assert _rows(mr, "k_prep") == [[512, 256]]
        grid(7, (0, 0, 0))  # 343 leaves: its own candidates
        assert sorted(_rows(mr, "k_prep")) == [[256, 128], [512, 256]]
        grid(2, (1, 1, 1))
        assert sorted(_rows(mr, "k_prep")) == [[256, 128], [512, 256], [512, 256]]
        assert len(_rows(mr, "k_merge")) == 2
        for order in (0, 2):
            small.set_diffusion(1e-3 if order else 0.0, order)
            small.rhs_advect(0, (0.5, 0.25, -0.5), 1, mr.WENOZ5)
        small.sync()
        assert len(_rows(mr, "k_fused")) == 2 and len(_rows(mr, "stage kernel")) == 2
    finally:
        mr.autotune_clear()
