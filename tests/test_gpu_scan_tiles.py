"""The cells' offsets on both sides of the sizes where their scan changes: one
tile and two, and up to 512 tiles of 1024 cells (a block adds up the tiles
before its own) and one past that (a scan of the tile sums comes first).
Offsets and the pair count are whole numbers: exact."""
import numpy as np
import pytest

from tests.gpu_util import _dev_array, torch_cuda
from tests.test_gpu_sort_sources import SEED, STEP, _species
from tests.test_gpu_small_binning import _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [5120, 5121, 255 * 1024 + 1, 512 * 1024, 512 * 1024 + 1, 600 * 1024 - 1])
def test_offsets(cells):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    rng = np.random.default_rng(cells)
    n = 100_000
    # most cells empty, and the last ones not
    e, g = (_species(rng, np.bincount(np.minimum(rng.integers(0, cells + 64, n), cells - 1), minlength=cells), "moved")
            for _ in range(2))
    ctx = cg.compton_init(cells, n, 1.0, 0.05, SEED)
    try:
        ein, gin = _dev(cg, torch, e), _dev(cg, torch, g)
        eo, go = cg.Species.empty_like(ein), cg.Species.empty_like(gin)
        for _ in range(2):
            pairs = cg.compton_bin_pairs(ctx, ein, gin, eo, go, STEP)
            assert cg.compton_check(ctx) == cg.COMPTON_OK
            counts = []
            for d, off in ((e, pairs.off_e_dev), (g, pairs.off_g_dev)):
                counts.append(np.bincount(d["cell"], minlength=cells))
                assert np.array_equal(_dev_array(torch, off, cells + 1), np.concatenate([[0], np.cumsum(counts[-1])]))
            assert _dev_array(torch, pairs.n_pairs_dev, 2).view(np.int64)[0] == np.minimum(*counts).sum()
    finally:
        cg.compton_destroy(ctx)
