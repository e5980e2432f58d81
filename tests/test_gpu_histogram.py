"""The histogram of cell indices and its order check, where runs of equal indices
begin and end at the edges of a lane's four positions, of a warp's 128 and of
its stretch; arrays that end inside them; indices out of range, at the start, the
end and inside runs; an index array off the 16-byte boundary.  Offsets are whole
numbers: exact.  (More than 4096 cells, so that no call is a small one.)"""
import numpy as np
import pytest

from tests.gpu_util import _dev_array, torch_cuda
from tests.test_gpu_sort_sources import SEED, STEP

pytestmark = pytest.mark.gpu
CELLS = 5000


def _cells(rng, n, run, kind):
    # runs of `run` positions, cell after cell and round again (no cell gets thousands)
    c = (rng.permutation(CELLS) if kind == "any" else np.arange(CELLS))[np.arange(n) // run % CELLS].astype(np.int32)
    if kind == "bad" and n > 8:
        c[[0, 3, 4, n // 2, n - 2, n - 1]] = (-1, CELLS, 1 << 30, -(1 << 31), CELLS, -1)
    return c


@pytest.mark.parametrize("kind", ["cells", "any", "bad"])
@pytest.mark.parametrize("n,run,shift", [(1, 1, 0), (3, 1, 0), (127, 4, 0), (128, 128, 0), (129, 64, 0), (131, 3, 1),
                                         (4096, 4, 0), (4097, 5, 3), (100_003, 63, 2), (1_300_001, 129, 0),
                                         (1_300_001, 1, 1)])
def test_counts(n, run, shift, kind):
    import paper_2206_02937_gb300 as cg
    torch = torch_cuda()
    cg.build()
    rng = np.random.default_rng(n + run)
    cells = [_cells(rng, n, run, kind), _cells(rng, n, run + 1, kind)]
    ctx = cg.compton_init(CELLS, n, 1.0, 0.05, SEED)
    try:
        species = []
        for c in cells:
            buf = torch.zeros(n + shift, dtype=torch.int32, device="cuda")
            buf[shift:] = torch.from_numpy(c).cuda()
            u = [torch.rand(n, device="cuda") for _ in range(3)]
            species.append(cg.Species(*u, buf[shift:], torch.arange(n, dtype=torch.int32, device="cuda")))
        out = [cg.Species.empty_like(s) for s in species]
        pairs = cg.compton_bin_pairs(ctx, *species, *out, STEP)
        ok = [(c >= 0) & (c < CELLS) for c in cells]
        assert cg.compton_check(ctx) == (cg.COMPTON_OK if all(o.all() for o in ok) else cg.COMPTON_ERANGE)
        for c, o, off in zip(cells, ok, (pairs.off_e_dev, pairs.off_g_dev)):
            want = np.concatenate([[0], np.cumsum(np.bincount(c[o], minlength=CELLS))])
            assert np.array_equal(_dev_array(torch, off, CELLS + 1), want)
    finally:
        cg.compton_destroy(ctx)
